// The EUVAC band sums S0 = sum_j B_j Phi_j e^{-Phi_j k} and S1 = sum_j B_j Phi_j^2 e^{-Phi_j k} (S1 is minus
// dS0/dk) on the integer pipe.
//
// 37 exponentials per point are most of the heating's cost in FP64 (16 FP64 instructions per band, 64 issue
// cycles of a warp each). Here a band takes about 75 integer instructions: with t = 128 Phi k / ln2 = n + f,
// |f| <= 1/2, e^{-Phi k} = 2^-(n >> 7) W[n & 127] 2^{-f/128}, where W[i] = 2^{-i/128} is a table and
// 1 - 2^{-f/128} a Taylor polynomial of degree 5, all in 57-bit fixed point (absolute error of the
// exponential below 2^-56, checked against 60-digit arithmetic). t keeps 57 bits, as many as the FP64 product
// Phi k. The terms are positive and summed exactly; they share the exponent of the least attenuated band, so
// a strongly attenuated sum keeps its relative accuracy. Arguments outside the checked range (negative,
// NaN, larger than 2^27) take the FP64 loop.
#pragma once

#include "dg_fx.cuh"
#include "dg_math64.cuh"

namespace dg {

struct EuvFx {
  int n;
  double tscale;             // max phi * 128 / ln2
  double s0, s1;             // one absorber: max(B phi), max(B phi^2); four: max B max phi, max B max phi^2
  double B[40], phi[4][40];  // the bands themselves (FP64 loop)
  int2 xphi[4][40], xlow[4]; // phi / max phi, and each species' smallest
  int2 xb[40], xc[40];       // B phi and B phi^2 of the first species over their maxima
  int2 xB[40];               // B / max B
};
// host: tables of n bands (coefficients with exponent 57, split at 29)
inline void build_euv(int n, const double* B, const double (*phi)[40], int species, EuvFx* x) {
  auto top = [](double m) { return m > 0.0 ? m : 1.0; };
  double pm = 0.0, bm = 0.0, b0 = 0.0, c0 = 0.0;
  for (int j = 0; j < n; ++j) {
    bm = B[j] > bm ? B[j] : bm;
    for (int s = 0; s < species; ++s) pm = phi[s][j] > pm ? phi[s][j] : pm;
    b0 = B[j] * phi[0][j] > b0 ? B[j] * phi[0][j] : b0;
    c0 = B[j] * phi[0][j] * phi[0][j] > c0 ? B[j] * phi[0][j] * phi[0][j] : c0;
  }
  pm = top(pm);
  bm = top(bm);
  b0 = top(b0);
  c0 = top(c0);
  auto coef = [](long double v) { return fx_coef(v < 1.0L ? v : 1.0L - 0x1p-57L, 57, 29); };
  *x = EuvFx();
  x->n = n;
  x->tscale = (double)((long double)pm * 128.0L / 0.693147180559945309417232121458176568L);
  x->s0 = species == 1 ? b0 : bm * pm;
  x->s1 = species == 1 ? c0 : bm * pm * pm;
  for (int s = 0; s < 4; ++s) {
    double low = s < species && n > 0 ? phi[s][0] : 0.0;
    for (int j = 0; j < n; ++j) {
      x->phi[s][j] = s < species ? phi[s][j] : 0.0;
      x->xphi[s][j] = coef((long double)x->phi[s][j] / pm);
      // one absorber: bands it does not absorb do not count
      if (s < species && (species > 1 || phi[s][j] > 0.0) && (phi[s][j] < low || (species == 1 && low == 0.0)))
        low = phi[s][j];
    }
    x->xlow[s] = coef((long double)low / pm);
  }
  for (int j = 0; j < n; ++j) {
    x->B[j] = B[j];
    x->xB[j] = coef((long double)B[j] / bm);
    x->xb[j] = coef((long double)B[j] * phi[0][j] / b0);
    x->xc[j] = coef((long double)B[j] * phi[0][j] * phi[0][j] / c0);
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

__device__ __forceinline__ fx fx_ld(const int2* p) {
  const int2 v = __ldg(p);
  return {v.x, v.y};
}

// t = A K 2^-s (A of exponent 57): n = rint(t), f57 = (t - n) 2^57
__device__ __forceinline__ int euv_split(fx A, fx K, int s, long long& f57) {
  const long long R = fx_mul<28>(A, K);
  const int sn = min(s, 62);
  const long long n = (R + (1LL << (sn - 1))) >> sn;
  f57 = ((R - (n << sn)) << max(57 - s, 0)) >> max(s - 57, 0);
  return (int)n;
}

// NS = 1: Phi_j = phi_j of the first species; NS = 4: Phi_j = sum_s w[s] phi_sj
template <int NS>
__device__ __forceinline__ void euvac_sums(const EuvFx* __restrict__ X, const double w[4], double k, double& S0,
                                           double& S1) {
  double kk = k * X->tscale;
  bool ok = kk >= 0.0;
  fx ws[4];
  int ew = 1020;
  if constexpr (NS == 4) {
    int m = 0;
    for (int s = 0; s < 4; ++s) {
      ok = ok && w[s] >= 0.0;
      m = max(m, fx_mag(w[s]));
    }
    ok = ok && (m >> 20) >= 900 && (m >> 20) <= 1100;
    ew = m >> 20;
    for (int s = 0; s < 4; ++s) ws[s] = fx_split<28>(fx_from<55>(w[s], ew));
    kk *= __hiloint2double((ew + 3) << 20, 0);   // 2^(ew - 1020)
  }
  const int hk = __double2hiint(kk);
  ok = ok && hk < (1050 << 20);
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
  const int ek = max(hk >> 20, 963), s = 1079 - ek;
  const fx K = fx_split<28>(fx_from<57>(kk, ek));
  fx low = fx_ld(&X->xlow[0]);
  if constexpr (NS == 4) {
    fxacc a = fx_zero<28>();
    for (int q = 0; q < 4; ++q) fx_mac(a, fx_ld(&X->xlow[q]), ws[q]);
    low = fx_split<29>(fx_sum<28>(a));
  }
  long long f57;
  const int emin = euv_split(low, K, s, f57) >> 7;
  fxacc a0 = fx_zero<28>(), a1 = fx_zero<28>();
#pragma unroll 1
  for (int j = 0; j < X->n; ++j) {
    fx A = fx_ld(&X->xphi[0][j]), b, c;
    if constexpr (NS == 4) {
      fxacc a = fx_zero<28>();
      fx_mac(a, A, ws[0]);
#pragma unroll
      for (int q = 1; q < 4; ++q) fx_mac(a, fx_ld(&X->xphi[q][j]), ws[q]);
      const long long Ai = fx_sum<28>(a);
      A = fx_split<29>(Ai);
      const fx Ah = fx_split<28>(Ai);
      const long long bi = fx_mul<28>(fx_ld(&X->xB[j]), Ah);
      b = fx_split<29>(bi);
      c = fx_split<29>(fx_mul<28>(b, Ah));
    } else {
      b = fx_ld(&X->xb[j]);
      c = fx_ld(&X->xc[j]);
    }
    const int n = euv_split(A, K, s, f57);
    // g = 1 - 2^{-f/128}, Horner with 2^31 f; the leading terms with all 57 bits of f
    const int u = (int)(f57 >> 26);
    const int p = 2581847 - (int)(((long long)u * 2796) >> 31);
    const int q = 1907106652 - (int)(((long long)u * p) >> 31);
    const long long h = 69240576462433397LL - (((long long)u * q) >> 15);
    const fx f = fx_split<29>(f57);
    const long long y = 99893036290645747LL - (fx_mul<28>(f, fx_split<28>(h)) >> 8);
    const long long g = fx_mul<28>(f, fx_split<28>(y));
    const long long W = kExp2Neg[n & 127];
    long long E = W - ((fx_mul<28>(fx_split<29>(W), fx_split<28>(g)) + 64) >> 7);
    E >>= min(max((n >> 7) - emin, 0), 63);
    const fx e = fx_split<28>(E);
    fx_mac(a0, b, e);
    fx_mac(a1, c, e);
  }
  const double z = emin > 900 ? 0.0 : __hiloint2double((1023 - 57 - emin) << 20, 0);
  const double sw = NS == 4 ? __hiloint2double((ew + 3) << 20, 0) : 1.0;
  S0 = (double)fx_sum<28>(a0) * (X->s0 * sw) * z;
  S1 = (double)fx_sum<28>(a1) * (X->s1 * sw * sw) * z;
}

}  // namespace dg
