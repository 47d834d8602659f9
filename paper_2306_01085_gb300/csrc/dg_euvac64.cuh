// The EUVAC band sums S0 = sum_j B_j Phi_j e^{-Phi_j k} and S1 = sum_j B_j Phi_j^2 e^{-Phi_j k} (S1 is minus
// dS0/dk) on the integer pipe.
//
// 37 exponentials per point are most of the heating's cost in FP64 (16 FP64 instructions per band, 64 issue
// cycles of a warp each). Here a band takes about 110 integer instructions: with t = 128 Phi k / ln2 = n + f,
// |f| <= 1/2, e^{-Phi k} = 2^-(n >> 7) W[n & 127] 2^{-f/128}, where W[i] = 2^{-i/128} is a table and
// 1 - 2^{-f/128} a Taylor polynomial of degree 5, in 57-bit fixed point (absolute error of the exponential
// below 2^-56). Bands differ by orders of magnitude in Phi, and at depth the weakest absorption carries the
// whole sum, so every band has its own exponents: Phi, B Phi, B Phi^2 and t are 58-bit mantissas with a
// binary exponent each (relative error a few 2^-57; four absorbers: their weighted sum likewise), and the
// sums' exponents follow the largest term met so far. Terms are positive. In units of 2^-53 (2 + tau), tau the
// mean optical depth of the bands that carry the sum, the relative errors stay below 0.46 (one absorber) and
// 0.64 (four) over 13 decades of k and fractions down to 1e-12; those of the FP64 loop reach 4 and 5.7. One
// exponent for all bands (that of the largest Phi) takes about 75 instructions and loses up to 1e-9 of S1 at depth.
// Negative or non-finite arguments, weights and fluxes, and zero or subnormal k, take the FP64 loop.
#pragma once

#include "dg_bits.cuh"
#include "dg_fx.cuh"

namespace dg {

// m 2^(e - 58) with 2^57 <= m < 2^58 (or m = 0), m = hi 2^29 + lo
struct alignas(16) EuvNum { int hi, lo, e, pad; };   // read by 16-byte loads
constexpr int EUV_NONE = -(1 << 20);   // exponent of zero

struct EuvFx {
  int n;
  int fixed;                 // every B and phi is finite and not negative
  double B[40], phi[4][40];  // the bands themselves (FP64 loop)
  EuvNum xphi[4][40];
  EuvNum xb[40], xc[40];     // one absorber: B phi and B phi^2; four: B and unused
};
static_assert(sizeof(EuvNum) == 16 && alignof(EuvFx) == 16, "band tables: one aligned 16-byte load per number");
inline EuvNum euv_num(long double v) {
  if (!(v > 0.0L)) return {0, 0, EUV_NONE, 0};
  int e;
  long long m = __builtin_llrintl(__builtin_ldexpl(__builtin_frexpl(v, &e), 58));
  if (m >> 58) {
    m >>= 1;
    ++e;
  }
  return {(int)(m >> 29), (int)(m & ((1 << 29) - 1)), e, 0};
}
// host: tables of n bands
inline void build_euv(int n, const double* B, const double (*phi)[40], int species, EuvFx* x) {
  *x = EuvFx();
  x->n = n;
  x->fixed = 1;
  for (int j = 0; j < n; ++j) {
    const long double b = B[j], f = phi[0][j];
    x->B[j] = B[j];
    if (!(B[j] >= 0.0 && B[j] < 1e100)) x->fixed = 0;
    for (int s = 0; s < species; ++s) {
      x->phi[s][j] = phi[s][j];
      x->xphi[s][j] = euv_num(phi[s][j]);
      if (!(phi[s][j] >= 0.0 && phi[s][j] < 1e100)) x->fixed = 0;
    }
    x->xb[j] = euv_num(species == 1 ? b * f : b);
    x->xc[j] = euv_num(b * f * f);
  }
}

// W[i] = 2^{-i/128} 2^57
static __device__ const long long kExp2Neg[128] = {
    0x200000000000000LL, 0x1fd3c22b8f71f11LL, 0x1fa7c1819e90d83LL, 0x1f7bfdad9cbe139LL,
    0x1f50765b6e45406LL, 0x1f252b376bba975LL, 0x1efa1bee615a277LL, 0x1ecf482d8e67f09LL,
    0x1ea4afa2a490d98LL, 0x1e7a51fbc74c835LL, 0x1e502ee78b3ff62LL, 0x1e264614f5a128aLL,
    0x1dfc97337b9b5ecLL, 0x1dd321f301b4605LL, 0x1da9e603db32857LL, 0x1d80e316c98397cLL,
    0x1d5818dcfba4872LL, 0x1d2f87080d89f19LL, 0x1d072d4a07897b9LL, 0x1cdf0b555dc3f9cLL,
    0x1cb720dcef90691LL, 0x1c8f6d9406e7b51LL, 0x1c67f12e57d14b5LL, 0x1c40ab5fffd07a7LL,
    0x1c199bdd85529c2LL, 0x1bf2c25bd71e088LL, 0x1bcc1e904bc1d22LL, 0x1ba5b030a106498LL,
    0x1b7f76f2fb5e46fLL, 0x1b59728de559399LL, 0x1b33a2b84f15fafLL, 0x1b0e07298db6659LL,
    0x1ae89f995ad3ad6LL, 0x1ac36bbfd3f379cLL, 0x1a9e6b5579fdbf4LL, 0x1a799e1330b3587LL,
    0x1a5503b23e255c9LL, 0x1a309bec4a2d336LL, 0x1a0c667b5de564bLL, 0x19e86319e323232LL,
    0x19c49182a3f0902LL, 0x19a0f170ca07b9cLL, 0x197d829fde4e4f9LL, 0x195a44cbc8520efLL,
    0x193737b0cdc5e4fLL, 0x19145b0b91ffc59LL, 0x18f1ae991577363LL, 0x18cf3216b5448bfLL,
    0x18ace5422aa0db6LL, 0x188ac7d98a66996LL, 0x1868d99b4492ec8LL, 0x18471a4623c7acdLL,
    0x182589994cce129LL, 0x180427543e1a11bLL, 0x17e2f336cf4e621LL, 0x17c1ed0130c1328LL,
    0x17a11473eb0186dLL, 0x1780694fde5d3f6LL, 0x175feb564267c8cLL, 0x173f9a48a58173cLL,
    0x171f75e8ec5f73eLL, 0x16ff7df9519483dLL, 0x16dfb23c651a2efLL, 0x16c012750bdabefLL,
    0x16a09e667f3bcc9LL, 0x168155d44ca9731LL, 0x166238825522249LL, 0x16434634ccc31fcLL,
    0x16247eb03a5584bLL, 0x1605e1b976dc08bLL, 0x15e76f15ad21487LL, 0x15c9268a5946b70LL,
    0x15ab07dd4854296LL, 0x158d12d497c7fd2LL, 0x156f4736b527da6LL, 0x1551a4ca5d920ecLL,
    0x15342b569d4f81eLL, 0x1516daa2cf6641cLL, 0x14f9b2769d2ca6bLL, 0x14dcb299fddd0d6LL,
    0x14bfdad5362a272LL, 0x14a32af0d7d3de6LL, 0x1486a2b5c13cd01LL, 0x146a41ed1d00577LL,
    0x144e086061892d0LL, 0x1431f5d950a896eLL, 0x14160a21f72e2a0LL, 0x13fa4504ac801baLL,
    0x13dea64c1234223LL, 0x13c32dc313a8e48LL, 0x13a7db34e59ff6fLL, 0x138cae6d05d8658LL,
    0x1371a7373aa9caaLL, 0x1356c55f929ff0dLL, 0x133c08b26416ff5LL, 0x132170fc4cd8313LL,
    0x1306fe0a31b7153LL, 0x12ecafa93e2f561LL, 0x12d285a6e4030b4LL, 0x12b87fd0dad9900LL,
    0x129e9df51fdee13LL, 0x1284dfe1f563809LL, 0x126b4565e27cdd2LL, 0x1251ce4fb2a63f3LL,
    0x12387a6e7562386LL, 0x121f49917ddc962LL, 0x12063b88628cd64LL, 0x11ed5022fcd91ccLL,
    0x11d4873168b9aa8LL, 0x11bbe084045cd3aLL, 0x11a35beb6fcb754LL, 0x118af9388c8de9cLL,
    0x1172b83c7d517aeLL, 0x115a98c8a58e512LL, 0x11429aaea92ddfbLL, 0x112abdc06c31cc0LL,
    0x111301d0125b50aLL, 0x10fb66affed31afLL, 0x10e3ec32d3d1a20LL, 0x10cc922b7247f74LL,
    0x10b5586cf9890f6LL, 0x109e3ecac6f3834LL, 0x10874518759bc81LL, 0x10706b29ddf6ddcLL,
    0x1059b0d31585744LL, 0x104315e86e7f84cLL, 0x102c9a3e778060fLL, 0x10163da9fb33357LL};

__device__ __forceinline__ EuvNum euv_ld(const EuvNum* p) {
#ifdef __CUDA_ARCH__
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return {v.x, v.y, v.z, 0};
#else
  return *p;
#endif
}
// mantissa and exponent of a positive normal double
__device__ __forceinline__ long long euv_mantissa(double x, int& e) {
  const uint64_t b = bits_of(x);
  e = (int)(b >> 52) - 1022;
  return (long long)((b & 0xfffffffffffffull) | 0x10000000000000ull) << 5;
}
// a mantissa of up to 59 bits back to 58
__device__ __forceinline__ void euv_norm(long long& m, int& e) {
  const int up = (int)(m >> 58);             // 0 or 1
  m >>= up;
  e += up;
}
// a 2^e += m 2^me, to 2^-56 of the larger; the sum holds 40 terms below 2^58 at half their unit
__device__ __forceinline__ void euv_add(long long& a, int& e, long long m, int me) {
  if (me > e) {
    a = ((a >> (min(me - e, 63) - 1)) + 1) >> 1;
    e = me;
  }
  a += ((m >> min(e - me, 62)) + 1) >> 1;
}
// x 2^e
__device__ __forceinline__ double euv_scale(double x, int e) {
  return e > -960 && e < 900 ? x * double_of((uint32_t)(e + 1023) << 20, 0u) : ldexp(x, e);
}

// NS = 1: Phi_j = phi_j of the first species; NS = 4: Phi_j = sum_s w[s] phi_sj
template <int NS>
__device__ __forceinline__ void euvac_sums(const EuvFx* __restrict__ X, const double w[4], double k, double& S0,
                                           double& S1) {
  auto usable = [](double x) { const int h = (int)(bits_of(x) >> 32); return h >= (200 << 20) && h < (1846 << 20); };
  bool ok = X->fixed != 0 && usable(k);
  if constexpr (NS == 4)
    for (int s = 0; s < 4; ++s) ok = ok && (w[s] == 0.0 || usable(w[s]));
  if (!ok) {
    S0 = S1 = 0.0;
#pragma unroll 1
    for (int j = 0; j < X->n; ++j) {
      double Phi = X->phi[0][j];
      if constexpr (NS == 4) Phi = fma(w[0], Phi, fma(w[1], X->phi[1][j], fma(w[2], X->phi[2][j], w[3] * X->phi[3][j])));
      const double a = (X->B[j] * Phi) * exp(-Phi * k);
      S0 += a;
      S1 = fma(Phi, a, S1);
    }
    return;
  }
  fx ws[4];
  int ew[4];
  if constexpr (NS == 4)
    for (int s = 0; s < 4; ++s) {
      const long long m = euv_mantissa(w[s], ew[s]);
      ws[s] = fx_split<28>(w[s] == 0.0 ? 0LL : m);
    }
  // K = k 128 / ln2
  int eK;
  long long Km = euv_mantissa(k, eK);
  Km = fx_mul<28>(fx_split<29>(207914267153817539LL), fx_split<28>(Km));
  eK += 7;
  euv_norm(Km, eK);
  const fx K = fx_split<28>(Km);
  long long a0 = 0, a1 = 0;
  int e0 = EUV_NONE, e1 = EUV_NONE;
#pragma unroll 1
  for (int j = 0; j < X->n; ++j) {
    EuvNum q = euv_ld(&X->xphi[0][j]);
    fx A{q.hi, q.lo}, b, c;
    int eA = q.e, eb, ec;
    if constexpr (NS == 4) {
      long long m[4];
      int em[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (s) q = euv_ld(&X->xphi[s][j]);
        m[s] = fx_mul<28>(fx{q.hi, q.lo}, ws[s]);
        em[s] = m[s] ? q.e + ew[s] - 1 : EUV_NONE;
      }
      eA = max(max(em[0], em[1]), max(em[2], em[3]));
      long long Am = 0;                      // below 2^61
#pragma unroll
      for (int s = 0; s < 4; ++s) Am += m[s] >> min(eA - em[s], 63);
      if (Am == 0) continue;
      const int up = max(6 - __clzll(Am), 0);
      Am >>= up;
      eA += up;
      A = fx_split<29>(Am);
      const fx Ah = fx_split<28>(Am);
      const EuvNum B = euv_ld(&X->xb[j]);
      long long x = fx_mul<28>(fx{B.hi, B.lo}, Ah);
      eb = B.e + eA - 1;
      euv_norm(x, eb);
      b = fx_split<29>(x);
      x = fx_mul<28>(b, Ah);
      ec = eb + eA - 1;
      euv_norm(x, ec);
      c = fx_split<29>(x);
    } else {
      q = euv_ld(&X->xb[j]);
      b = fx{q.hi, q.lo};
      eb = q.e;
      q = euv_ld(&X->xc[j]);
      c = fx{q.hi, q.lo};
      ec = q.e;
    }
    // t = R 2^-s = n + f57 2^-57
    const int s = 59 - eA - eK;
    if (s < 31 || b.hi == 0) continue;       // t of 2^26 and more: the attenuation is below the FP64 range
    const long long R = fx_mul<28>(A, K);
    const int sn = min(s, 62);
    const int n = (int)((R + (1LL << (sn - 1))) >> sn);
    const long long f57 = ((R - ((long long)n << sn)) << max(57 - s, 0)) >> min(max(s - 57, 0), 63);
    // g = 1 - 2^{-f/128}, Horner with 2^31 f; the leading terms with all 57 bits of f
    const int u = (int)(f57 >> 26);
    const int p = 2581847 - (int)(((long long)u * 2796) >> 31);
    const int r = 1907106652 - (int)(((long long)u * p) >> 31);
    const long long h = 69240576462433397LL - (((long long)u * r) >> 15);
    const fx f = fx_split<29>(f57);
    const long long y = 99893036290645747LL - (fx_mul<28>(f, fx_split<28>(h)) >> 8);
    const long long g = fx_mul<28>(f, fx_split<28>(y));
    const long long W = kExp2Neg[n & 127];
    const fx E = fx_split<28>(W - ((fx_mul<28>(fx_split<29>(W), fx_split<28>(g)) + 64) >> 7));
    const int d = n >> 7;
    euv_add(a0, e0, fx_mul<28>(b, E), eb - d);
    euv_add(a1, e1, fx_mul<28>(c, E), ec - d);
  }
  S0 = a0 ? euv_scale((double)a0, e0 - 57) : 0.0;
  S1 = a1 ? euv_scale((double)a1, e1 - 57) : 0.0;
}

}  // namespace dg
