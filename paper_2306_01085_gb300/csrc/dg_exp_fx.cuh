// Exponential, its pair e^x, e^-x, and powers of the pointwise physics in fixed point, without FP64 instructions.
//
// An FP64 instruction costs a warp 64 issue cycles of its scheduler on GB300, a 32 x 32 + 64 bit multiply-add
// about 2. The table-driven scheme of P. T. P. Tang (ACM TOMS 15, 1989, exponential; ACM TOMS 16, 1990,
// logarithm) with 128 entries is evaluated on 64-bit integers: the products that the result's last bits depend on
// are formed from 31-bit halves, the series beyond the quadratic term from the high halves alone. An argument is
// held at 2^-56 (exact from 2^-4 on), a reduced one at 2^-70 (logarithm: 2^-64, exact).
//   fx_exp, fx_exp_pm   |x| < 64; error below 0.65 ulp: rounding 0.5, argument 2^-57 and series 2^-58 relative
//   fx_power            u^a e^(-a v / 2) for 2^-40 <= u < 2^41, |v| < 64, 0 < a < 1; error below 1.2 ulp: the series of
//                       the logarithm adds 3 units of 2^-56, the product with a one
// against 10, 14 and 26 FP64 instructions. The same functions compile for the host, where they are tested.
#pragma once

#include "dg_bits.cuh"

namespace dg {

// 2^(j/128) 2^62
static __device__ const long long kExp2Fx[128] = {
    0x4000000000000000LL, 0x4058f6a7ecccd5b6LL, 0x40b268f9de0183baLL, 0x410c57a1b9fe12f6LL, 0x4166c34c5615d0ecLL,
    0x41c1aca777db771bLL, 0x421d1461d66f2023LL, 0x4278fb2b1bce0d15LL, 0x42d561b3e6243d8aLL, 0x433248adc91fdd02LL,
    0x438fb0cb4f468808LL, 0x43ed9abffb4c6bc9LL, 0x444c0740496d4294LL, 0x44aaf701b0c72feeLL, 0x450a6abaa4b77ecdLL,
    0x456a632296394492LL, 0x45cae0f1f545eb73LL, 0x462be4e23237a6efLL, 0x468d6fadbf2dd4f3LL, 0x46ef821011734e6bLL,
    0x47521cc5a2e6a9e0LL, 0x47b5408bf36472e2LL, 0x4818ee218a3358eeLL, 0x487d2645f7725895LL, 0x48e1e9b9d588e19bLL,
    0x4947393eca98fcd6LL, 0x49ad159789f37496LL, 0x4a137f87d58e025bLL, 0x4a7a77d47f7b84b1LL, 0x4ae1ff436b663ff7LL,
    0x4b4a169b900c2d00LL, 0x4bb2bea4f8bd5847LL, 0x4c1bf828c6dc54b8LL, 0x4c85c3f13360c4d5LL, 0x4cf022c9905bfd32LL,
    0x4d5b157e4a7fc325LL, 0x4dc69cdceaa72a9cLL, 0x4e32b9b417619617LL, 0x4e9f6cd3967fdba8LL, 0x4f0cb70c4ea39210LL,
    0x4f7a993048d088d7LL, 0x4fe91412b2006e83LL, 0x50582887dcb8a7e1LL, 0x50c7d76542a25b72LL, 0x513821818624b40cLL,
    0x51a907b474015dc9LL, 0x521a8ad704f3404fLL, 0x528cabc35f4f799dLL, 0x52ff6b54d8a89c75LL, 0x5372ca67f774358fLL,
    0x53e6c9da74b29ab5LL, 0x545b6a8b3d990704LL, 0x54d0ad5a753e077cLL, 0x5546932976483b15LL, 0x55bd1cdad49f699cLL,
    0x56344b525f1ff495LL, 0x56ac1f752150a563LL, 0x57249a29651adc07LL, 0x579dbc56b48521baLL, 0x581786e5db7022c2LL,
    0x5891fac0e95612c8LL, 0x590d18d3330c7f1eLL, 0x5988e20954889245LL, 0x5a05575132a5cc20LL, 0x5a827999fcef3242LL,
    0x5b0049d42f6afbb6LL, 0x5b7ec8f19468bbc9LL, 0x5bfdf7e546520f3eLL, 0x5c7dd7a3b17dcf75LL, 0x5cfe69229605cef5LL,
    0x5d7fad59099f22feLL, 0x5e01a53f7974fd86LL, 0x5e8451cfac061b5fLL, 0x5f07b404c304c9f1LL, 0x5f8bccdb3d398841LL,
    0x60109d50f86846d8LL, 0x6096266533384a2bLL, 0x611c69188f1eb339LL, 0x61a3666d124bb204LL, 0x622b1f66299a6599LL,
    0x62b39508aa836d6fLL, 0x633cc85ad5122fbdLL, 0x63c6ba6455dcd8aeLL, 0x64516c2e47ff1623LL, 0x64dcdec3371793d1LL,
    0x6569132f21483ba7LL, 0x65f60a7f79393e2eLL, 0x6683c5c3281ee6e9LL, 0x6712460a8fc24072LL, 0x67a18c678c8c8c61LL,
    0x683199ed779592caLL, 0x68c26fb128b4cd63LL, 0x69540ec8f895722dLL, 0x69e6784cc2cd61bdLL, 0x6a79ad55e7f6fd10LL,
    0x6b0daeff4fcde703LL, 0x6ba27e656b4eb57aLL, 0x6c381ca636d99642LL, 0x6cce8ae13c57ebdbLL, 0x6d65ca379564e639LL,
    0x6dfddbcbed791babLL, 0x6e96c0c284192610LL, 0x6f307a412f074892LL, 0x6fcb096f5c782210LL, 0x70666f76154a7089LL,
    0x7102ad7fff41e9b4LL, 0x719fc4b95f452d29LL, 0x723db6501b9ed447LL, 0x72dc8373be41a454LL, 0x737c2d55770fe711LL,
    0x741cb5281e25ee34LL, 0x74be1c203627c62bLL, 0x75606373ee921c97LL, 0x76038c5b260e5eeeLL, 0x76a7980f6cca15c2LL,
    0x774c87cc06d1812eLL, 0x77f25ccdee6d7ae6LL, 0x78991853d684a285LL, 0x7940bb9e2cffd89dLL, 0x79e947ef1d320d2dLL,
    0x7a92be8a92436616LL, 0x7b3d20b6399fc237LL, 0x7be86fb985689ddcLL, 0x7c94acddaeea5d3aLL, 0x7d41d96db915019dLL,
    0x7deff6b672f84e24LL, 0x7e9f06067a4360baLL, 0x7f4f08ae3dc7c426LL,
};
// k_j / 4096 close to 1 / (1 + (j + 1/2) / 128) and -log of it, 2^57
struct LogFx { long long l; int k; };
static __device__ const LogFx kLogFx[128] = {
    {0x20100ab2b1167LL, 4080}, {0x5e8b20b884b19LL, 4049}, {0x9d8125bc62b35LL, 4018}, {0xdcf4013f0c8c7LL, 3987},
    {0x11ad398c6cd588LL, 3957}, {0x1592bbc15215c9LL, 3927}, {0x195e430f8ce45eLL, 3898}, {0x1d310ba20455a1LL, 3869},
    {0x20e9106c52c816LL, 3841}, {0x24a80c5e15282eLL, 3813}, {0x286e19c056fbd0LL, 3785}, {0x2c187174f328b9LL, 3758},
    {0x2fa66d0f852791LL, 3732}, {0x335e249ac98c4cLL, 3705}, {0x36f93065eb0034LL, 3679}, {0x3a76e7e6fc3f35LL, 3654},
    {0x3e1ee19bb325c6LL, 3628}, {0x41a934749b1796LL, 3603}, {0x451536254dd071LL, 3579}, {0x48abfcb76f65c4LL, 3554},
    {0x4bfefca699916eLL, 3531}, {0x4f7ceac4d417daLL, 3507}, {0x52db5bfbf88a91LL, 3484}, {0x563f839318bab8LL, 3461},
    {0x59a9750a8eb4d1LL, 3438}, {0x5cf2e41d3f4533LL, 3416}, {0x606862d08814d3LL, 3393}, {0x639623aeb0b6fbLL, 3372},
    {0x66f018bc9bf0eaLL, 3350}, {0x6a2853ffb99af6LL, 3329}, {0x6d65c6884eb36aLL, 3308}, {0x70a881584164feLL, 3287},
    {0x73c8757b2ea993LL, 3267}, {0x7715b2b914bd67LL, 3246}, {0x7a3fc988aeaf1cLL, 3226}, {0x7d46098b0e0208LL, 3207},
    {0x807a0238639922LL, 3187}, {0x8389c3026ac314LL, 3168}, {0x869e3ac366af21LL, 3149}, {0x89b7781741485fLL, 3130},
    {0x8cab69dcde17d3LL, 3112}, {0x8fce1cfba62abbLL, 3093}, {0x92cb2086fcb1d0LL, 3075}, {0x95cca1d835ebb0LL, 3057},
    {0x98d2ae83d42c85LL, 3039}, {0x9bb1f32322a316LL, 3022}, {0x9e955d9d9da6f7LL, 3005}, {0xa1a8d99ba1f5c6LL, 2987},
    {0xa494f46da73721LL, 2970}, {0xa758f9b5838c20LL, 2954}, {0xaa4d762ef7c40bLL, 2937}, {0xad19759727565bLL, 2921},
    {0xafe963c63c4141LL, 2905}, {0xb2bd4bdb26a1b6LL, 2889}, {0xb5953924456c75LL, 2873}, {0xb871372075afd3LL, 2857},
    {0xbb2330cbf1b6f0LL, 2842}, {0xbe073093c2e39bLL, 2826}, {0xc0c0c101d7e400LL, 2811}, {0xc37e0ce828a474LL, 2796},
    {0xc63f1e8e40597cLL, 2781}, {0xc8d49f8fa53d44LL, 2767}, {0xcb9d1a189ab56eLL, 2752}, {0xce39982ea3f5d9LL, 2738},
    {0xd0d9838fbafed3LL, 2724}, {0xd3ad4544e46192LL, 2709}, {0xd623c681028378LL, 2696}, {0xd8ce3092d37b57LL, 2682},
    {0xdb7c2cf477b1d0LL, 2668}, {0xddfc64af244dfaLL, 2655}, {0xe0b15faef91f25LL, 2641}, {0xe33827200b7fc2LL, 2628},
    {0xe5c223a85ccca8LL, 2615}, {0xe84f5d7714eebcLL, 2602}, {0xeadfdcdad738f8LL, 2589}, {0xed73aa4264b0aeLL, 2576},
    {0xefd7acef460aeaLL, 2564}, {0xf271ed76edafb0LL, 2551}, {0xf4dbf330840ad2LL, 2539}, {0xf748e673069245LL, 2527},
    {0xf9b8ce612e4d81LL, 2515}, {0xfc2bb237ea3111LL, 2503}, {0xfea1994ee01b25LL, 2491}, {0x1011a8b18f0ed6aLL, 2479},
    {0x103968f24bfdb68LL, 2467}, {0x105e04c1aa2c060LL, 2456}, {0x1086248abc4f3abLL, 2444}, {0x10ab18bf5823c36LL, 2433},
    {0x10d037d237f463cLL, 2422}, {0x10f5822744fca29LL, 2411}, {0x111e62229bbf49bLL, 2399}, {0x11409a2e6c81da1LL, 2389},
    {0x116668af4dd395aLL, 2378}, {0x118c640ff75f05cLL, 2367}, {0x11b28cbb6ec93e9LL, 2356}, {0x11d5650035a98acLL, 2346},
    {0x11fbe551db43c13LL, 2335}, {0x121f0dfc65ceebeLL, 2325}, {0x12425d72bd380fdLL, 2315}, {0x1265d40adef0b85LL, 2305},
    {0x128d041990b0eabLL, 2294}, {0x12b0cdfbf7ad02aLL, 2284}, {0x12d1260ad99c763LL, 2275}, {0x12f53c9cc594222LL, 2265},
    {0x13197c0fa80e6a2LL, 2255}, {0x133de4c086c409fLL, 2245}, {0x135eccf0ac61cfcLL, 2236}, {0x1383850278cfd8aLL, 2226},
    {0x13a4b53f86cb2e7LL, 2217}, {0x13c6080c36bfb52LL, 2208}, {0x13eb37978b85b56LL, 2198}, {0x140cd448ff6dd67LL, 2189},
    {0x142e946de080bf0LL, 2180}, {0x1450785145cafd8LL, 2171}, {0x1472803f35eaadcLL, 2162}, {0x1494ac84ab0ed2bLL, 2153},
    {0x14b6fd6f970c1f7LL, 2144}, {0x14d59d43fdaba1fLL, 2136}, {0x14f8343f9cb678eLL, 2127}, {0x151af0c774a2d01LL, 2118},
    {0x1539f107e1d309dLL, 2110}, {0x155cf55c5a5437cLL, 2101}, {0x157c35f3490183cLL, 2093}, {0x159b952dcd3e282LL, 2085},
    {0x15bf053a48690e0LL, 2076}, {0x15dea65985a34fdLL, 2068}, {0x15fe66db2289921LL, 2060}, {0x161e46fda56466cLL, 2052},
};

// round(x 2^(1084 - TOP)) for a biased exponent of at most TOP
template <int TOP>
__host__ __device__ __forceinline__ long long fx_fixed(double x) {
  const uint64_t b = bits_of(x);
  const int hi = (int)(b >> 32), d = TOP - ((hi >> 20) & 0x7ff);
  const uint64_t m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
  const long long X = (long long)((((m << 10) >> (d < 63 ? d : 63)) + 1) >> 1);
  return hi < 0 ? -X : X;
}
__host__ __device__ __forceinline__ int biased_exp(double x) { return (int)(bits_of(x) >> 52) & 0x7ff; }

// x = X 2^-56 = n ln2 / 128 + r 2^-70
__host__ __device__ __forceinline__ long long fx_exp_reduce(long long X, int& n) {
  n = (int)(((long long)(int)(X >> 32) * 774541002 + (1LL << 45)) >> 46);
  return ((X - n * 390207173010335LL) << 14) - (((long long)n * -829548) >> 10);
}
// 2^(n / 128) (1 + p 2^-70), rounded; T = kExp2Fx[n & 127]
__host__ __device__ __forceinline__ double fx_exp_scale(int n, long long T, long long p) {
  const int Th = (int)(T >> 32), Tl = (int)((T & 0xffffffffLL) >> 1), ph = (int)(p >> 31), pl = (int)(p & 0x7fffffff);
  long long v = T + (((long long)Th * ph + (((long long)Tl * ph + (long long)Th * pl) >> 31)) >> 7);
  int e = (n >> 7) + 1022;
  if (v < (1LL << 62)) {
    v <<= 1;
    --e;
  }
  const uint64_t b = ((uint64_t)e << 52) + ((uint64_t)(v + 512) >> 10);   // the leading bit adds 1 to e
  return double_of((uint32_t)(b >> 32), (uint32_t)b);
}
// odd = r + r^3 / 6 + r^5 / 120, even = r^2 / 2 + r^4 / 24 at 2^-70
__host__ __device__ __forceinline__ void fx_exp_series(long long r, long long& odd, long long& even) {
  const int rh = (int)(r >> 31), rl = (int)(r & 0x7fffffff);
  const long long r2 = (long long)rh * rh + (((long long)rh * rl) >> 30);        // 2^-78
  const int r2h = (int)(r2 >> 31);                                              // 2^-47
  const int c = 1431655765 + (int)(((long long)r2h * 1145324612) >> 51);         // 1/6 + r^2 / 120, 2^-33
  const int t = (int)(((long long)rh * c) >> 31);                               // r / 6 + r^3 / 120, 2^-41
  const int w = (int)(((long long)r2h * 1431655765) >> 35);                      // r^2 / 24, 2^-47
  odd = r + (((long long)r2h * t) >> 18);
  even = (r2 >> 9) + (((long long)r2h * w) >> 24);
}
__device__ __forceinline__ double fx_exp_fixed(long long X) {
  int n;
  long long odd, even;
  fx_exp_series(fx_exp_reduce(X, n), odd, even);
  return fx_exp_scale(n, kExp2Fx[n & 127], odd + even);
}
__host__ __device__ __forceinline__ bool fx_exp_range(double x) { return biased_exp(x) <= 1028; }
__device__ __forceinline__ double fx_exp(double x) { return fx_exp_fixed(fx_fixed<1028>(x)); }
__device__ __forceinline__ void fx_exp_pm(double x, double& ep, double& em) {
  int n;
  long long odd, even;
  fx_exp_series(fx_exp_reduce(fx_fixed<1028>(x), n), odd, even);
  ep = fx_exp_scale(n, kExp2Fx[n & 127], even + odd);
  em = fx_exp_scale(-n, kExp2Fx[-n & 127], even - odd);
}

// log u at 2^-57
__device__ __forceinline__ long long fx_log(double u) {
  const uint64_t b = bits_of(u);
  const LogFx c = kLogFx[(int)(b >> 45) & 127];
  const int e = (int)(b >> 52) - 1023;
  // (1 + r) 2^64 = m k modulo 2^64
  const long long r = (long long)(((b & 0xfffffffffffffull) | 0x10000000000000ull) * (uint64_t)c.k);
  const int rh = (int)(r >> 26), rl = (int)(r & 0x3ffffff);                     // 2^-38, 2^-64
  const long long r2 = (long long)rh * rh + (((long long)rh * rl) >> 25);        // 2^-76
  int t = 1431655765 - (int)(((long long)rh * 1227133513) >> 38);                // 1/6 - r / 7, 2^-33
  t = 1717986918 - (int)(((long long)rh * t) >> 38);                            // 1/5 - ..., 2^-33
  t = 1073741824 - (int)(((long long)rh * t) >> 39);                            // 1/4 - ..., 2^-32
  t = 1431655765 - (int)(((long long)rh * t) >> 38);                            // 1/3 - ..., 2^-32
  t = (int)(((long long)rh * t) >> 30);                                         // r / 3 - ..., 2^-40
  const long long s = r - (r2 >> 13) + (((long long)(int)(r2 >> 30) * t) >> 22);
  return e * 99893036290645747LL + (((long long)e * 1469302631LL) >> 32) + c.l + (s >> 7);
}
__host__ __device__ __forceinline__ bool fx_power_range(double a, double u, double v) {
  const int h = (int)(bits_of(u) >> 52);
  return h >= 983 && h <= 1063 && biased_exp(v) <= 1028 && a > 0.0 && a < 1.0;
}
// exp(a (log u - v / 2))
__device__ __forceinline__ double fx_power(double a, double u, double v) {
  const long long D = fx_log(u) - fx_fixed<1028>(v);                            // v / 2 at 2^-57
  const long long A = fx_fixed<1022>(a);                                        // 2^-62
  const int Ah = (int)(A >> 31), Al = (int)(A & 0x7fffffff), Dh = (int)(D >> 32), Dl = (int)((D & 0xffffffffLL) >> 1);
  return fx_exp_fixed((long long)Ah * Dh + (((long long)Ah * Dl + (long long)Al * Dh) >> 31));
}

}  // namespace dg
