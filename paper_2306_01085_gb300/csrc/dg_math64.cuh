// FP64 exponentials and powers of the pointwise physics with few FP64 instructions.
//
// GB300 has 2 FP64 lanes per SM, so an FP64 instruction costs a warp 64 issue cycles of its scheduler
// while table look-ups and integer instructions are nearly free beside it. These functions follow the
// table-driven scheme of P. T. P. Tang (ACM TOMS 15, 1989, exponential; ACM TOMS 16, 1990, logarithm):
// a 128-entry table carries most of the argument and a short Taylor polynomial the rest.
//   exp_fast      10 FP64 instructions, error below 1 ulp (|x| <= 700; outside: CUDA's exp)
//   exp_pm_fast   e^x and e^-x together in 14
//   log_fast      11 (positive normal arguments), absolute error below 1e-16 (1 + |log x|)
//   recip_fast     4, from the hardware's reciprocal seed and two Newton steps, error below 1 ulp
// Their special cases (Inf, NaN, zero, negative, subnormal) go to the CUDA functions.
#pragma once

#include <cuda_runtime.h>

namespace dg {

// 2^(j/128)
static __device__ const double kExp2[128] = {
    0x1.0000000000000p+0, 0x1.0163da9fb3335p+0, 0x1.02c9a3e778061p+0, 0x1.04315e86e7f85p+0,
    0x1.059b0d3158574p+0, 0x1.0706b29ddf6dep+0, 0x1.0874518759bc8p+0, 0x1.09e3ecac6f383p+0,
    0x1.0b5586cf9890fp+0, 0x1.0cc922b7247f7p+0, 0x1.0e3ec32d3d1a2p+0, 0x1.0fb66affed31bp+0,
    0x1.11301d0125b51p+0, 0x1.12abdc06c31ccp+0, 0x1.1429aaea92de0p+0, 0x1.15a98c8a58e51p+0,
    0x1.172b83c7d517bp+0, 0x1.18af9388c8deap+0, 0x1.1a35beb6fcb75p+0, 0x1.1bbe084045cd4p+0,
    0x1.1d4873168b9aap+0, 0x1.1ed5022fcd91dp+0, 0x1.2063b88628cd6p+0, 0x1.21f49917ddc96p+0,
    0x1.2387a6e756238p+0, 0x1.251ce4fb2a63fp+0, 0x1.26b4565e27cddp+0, 0x1.284dfe1f56381p+0,
    0x1.29e9df51fdee1p+0, 0x1.2b87fd0dad990p+0, 0x1.2d285a6e4030bp+0, 0x1.2ecafa93e2f56p+0,
    0x1.306fe0a31b715p+0, 0x1.32170fc4cd831p+0, 0x1.33c08b26416ffp+0, 0x1.356c55f929ff1p+0,
    0x1.371a7373aa9cbp+0, 0x1.38cae6d05d866p+0, 0x1.3a7db34e59ff7p+0, 0x1.3c32dc313a8e5p+0,
    0x1.3dea64c123422p+0, 0x1.3fa4504ac801cp+0, 0x1.4160a21f72e2ap+0, 0x1.431f5d950a897p+0,
    0x1.44e086061892dp+0, 0x1.46a41ed1d0057p+0, 0x1.486a2b5c13cd0p+0, 0x1.4a32af0d7d3dep+0,
    0x1.4bfdad5362a27p+0, 0x1.4dcb299fddd0dp+0, 0x1.4f9b2769d2ca7p+0, 0x1.516daa2cf6642p+0,
    0x1.5342b569d4f82p+0, 0x1.551a4ca5d920fp+0, 0x1.56f4736b527dap+0, 0x1.58d12d497c7fdp+0,
    0x1.5ab07dd485429p+0, 0x1.5c9268a5946b7p+0, 0x1.5e76f15ad2148p+0, 0x1.605e1b976dc09p+0,
    0x1.6247eb03a5585p+0, 0x1.6434634ccc320p+0, 0x1.6623882552225p+0, 0x1.68155d44ca973p+0,
    0x1.6a09e667f3bcdp+0, 0x1.6c012750bdabfp+0, 0x1.6dfb23c651a2fp+0, 0x1.6ff7df9519484p+0,
    0x1.71f75e8ec5f74p+0, 0x1.73f9a48a58174p+0, 0x1.75feb564267c9p+0, 0x1.780694fde5d3fp+0,
    0x1.7a11473eb0187p+0, 0x1.7c1ed0130c132p+0, 0x1.7e2f336cf4e62p+0, 0x1.80427543e1a12p+0,
    0x1.82589994cce13p+0, 0x1.8471a4623c7adp+0, 0x1.868d99b4492edp+0, 0x1.88ac7d98a6699p+0,
    0x1.8ace5422aa0dbp+0, 0x1.8cf3216b5448cp+0, 0x1.8f1ae99157736p+0, 0x1.9145b0b91ffc6p+0,
    0x1.93737b0cdc5e5p+0, 0x1.95a44cbc8520fp+0, 0x1.97d829fde4e50p+0, 0x1.9a0f170ca07bap+0,
    0x1.9c49182a3f090p+0, 0x1.9e86319e32323p+0, 0x1.a0c667b5de565p+0, 0x1.a309bec4a2d33p+0,
    0x1.a5503b23e255dp+0, 0x1.a799e1330b358p+0, 0x1.a9e6b5579fdbfp+0, 0x1.ac36bbfd3f37ap+0,
    0x1.ae89f995ad3adp+0, 0x1.b0e07298db666p+0, 0x1.b33a2b84f15fbp+0, 0x1.b59728de5593ap+0,
    0x1.b7f76f2fb5e47p+0, 0x1.ba5b030a1064ap+0, 0x1.bcc1e904bc1d2p+0, 0x1.bf2c25bd71e09p+0,
    0x1.c199bdd85529cp+0, 0x1.c40ab5fffd07ap+0, 0x1.c67f12e57d14bp+0, 0x1.c8f6d9406e7b5p+0,
    0x1.cb720dcef9069p+0, 0x1.cdf0b555dc3fap+0, 0x1.d072d4a07897cp+0, 0x1.d2f87080d89f2p+0,
    0x1.d5818dcfba487p+0, 0x1.d80e316c98398p+0, 0x1.da9e603db3285p+0, 0x1.dd321f301b460p+0,
    0x1.dfc97337b9b5fp+0, 0x1.e264614f5a129p+0, 0x1.e502ee78b3ff6p+0, 0x1.e7a51fbc74c83p+0,
    0x1.ea4afa2a490dap+0, 0x1.ecf482d8e67f1p+0, 0x1.efa1bee615a27p+0, 0x1.f252b376bba97p+0,
    0x1.f50765b6e4540p+0, 0x1.f7bfdad9cbe14p+0, 0x1.fa7c1819e90d8p+0, 0x1.fd3c22b8f71f1p+0,
};
// c_j close to 1 / (1 + (j + 1/2) / 128), twelve significant bits, and -log(c_j)
static __device__ const double2 kLog[128] = {
    {0x1.fe00000000000p-1, 0x1.0080559588b35p-8}, {0x1.fa20000000000p-1, 0x1.7a2c82e212c65p-7},
    {0x1.f640000000000p-1, 0x1.3b024b78c5669p-6}, {0x1.f260000000000p-1, 0x1.b9e8027e1918ep-6},
    {0x1.eea0000000000p-1, 0x1.1ad398c6cd588p-5}, {0x1.eae0000000000p-1, 0x1.592bbc15215c9p-5},
    {0x1.e740000000000p-1, 0x1.95e430f8ce45ep-5}, {0x1.e3a0000000000p-1, 0x1.d310ba20455a1p-5},
    {0x1.e020000000000p-1, 0x1.074883629640bp-4}, {0x1.dca0000000000p-1, 0x1.254062f0a9417p-4},
    {0x1.d920000000000p-1, 0x1.4370ce02b7de8p-4}, {0x1.d5c0000000000p-1, 0x1.60c38ba79945dp-4},
    {0x1.d280000000000p-1, 0x1.7d33687c293c9p-4}, {0x1.cf20000000000p-1, 0x1.9af124d64c626p-4},
    {0x1.cbe0000000000p-1, 0x1.b7c9832f5801ap-4}, {0x1.c8c0000000000p-1, 0x1.d3b73f37e1f9bp-4},
    {0x1.c580000000000p-1, 0x1.f0f70cdd992e3p-4}, {0x1.c260000000000p-1, 0x1.06a4d1d26c5e6p-3},
    {0x1.bf60000000000p-1, 0x1.1454d8953741cp-3}, {0x1.bc40000000000p-1, 0x1.22aff2ddbd971p-3},
    {0x1.b960000000000p-1, 0x1.2ffbf29a6645cp-3}, {0x1.b660000000000p-1, 0x1.3df3ab13505f7p-3},
    {0x1.b380000000000p-1, 0x1.4b6d6fefe22a4p-3}, {0x1.b0a0000000000p-1, 0x1.58fe0e4c62eaep-3},
    {0x1.adc0000000000p-1, 0x1.66a5d42a3ad34p-3}, {0x1.ab00000000000p-1, 0x1.73cb9074fd14dp-3},
    {0x1.a820000000000p-1, 0x1.81a18b4220535p-3}, {0x1.a580000000000p-1, 0x1.8e588ebac2dbfp-3},
    {0x1.a2c0000000000p-1, 0x1.9bc062f26fc3ap-3}, {0x1.a020000000000p-1, 0x1.a8a14ffee66bdp-3},
    {0x1.9d80000000000p-1, 0x1.b5971a213acdbp-3}, {0x1.9ae0000000000p-1, 0x1.c2a205610593fp-3},
    {0x1.9860000000000p-1, 0x1.cf21d5ecbaa65p-3}, {0x1.95c0000000000p-1, 0x1.dc56cae452f5ap-3},
    {0x1.9340000000000p-1, 0x1.e8ff2622babc7p-3}, {0x1.90e0000000000p-1, 0x1.f518262c38082p-3},
    {0x1.8e60000000000p-1, 0x1.00f40470c7324p-2}, {0x1.8c00000000000p-1, 0x1.07138604d5862p-2},
    {0x1.89a0000000000p-1, 0x1.0d3c7586cd5e4p-2}, {0x1.8740000000000p-1, 0x1.136ef02e8290cp-2},
    {0x1.8500000000000p-1, 0x1.1956d3b9bc2fap-2}, {0x1.82a0000000000p-1, 0x1.1f9c39f74c557p-2},
    {0x1.8060000000000p-1, 0x1.2596410df963ap-2}, {0x1.7e20000000000p-1, 0x1.2b9943b06bd76p-2},
    {0x1.7be0000000000p-1, 0x1.31a55d07a8591p-2}, {0x1.79c0000000000p-1, 0x1.3763e64645463p-2},
    {0x1.77a0000000000p-1, 0x1.3d2abb3b3b4dfp-2}, {0x1.7560000000000p-1, 0x1.4351b33743eb9p-2},
    {0x1.7340000000000p-1, 0x1.4929e8db4e6e4p-2}, {0x1.7140000000000p-1, 0x1.4eb1f36b07184p-2},
    {0x1.6f20000000000p-1, 0x1.549aec5def881p-2}, {0x1.6d20000000000p-1, 0x1.5a32eb2e4eacbp-2},
    {0x1.6b20000000000p-1, 0x1.5fd2c78c78828p-2}, {0x1.6920000000000p-1, 0x1.657a97b64d437p-2},
    {0x1.6720000000000p-1, 0x1.6b2a72488ad8fp-2}, {0x1.6520000000000p-1, 0x1.70e26e40eb5fap-2},
    {0x1.6340000000000p-1, 0x1.76466197e36dep-2}, {0x1.6140000000000p-1, 0x1.7c0e612785c73p-2},
    {0x1.5f60000000000p-1, 0x1.81818203afc80p-2}, {0x1.5d80000000000p-1, 0x1.86fc19d05148ep-2},
    {0x1.5ba0000000000p-1, 0x1.8c7e3d1c80b30p-2}, {0x1.59e0000000000p-1, 0x1.91a93f1f4a7a8p-2},
    {0x1.5800000000000p-1, 0x1.973a3431356aep-2}, {0x1.5640000000000p-1, 0x1.9c73305d47ebbp-2},
    {0x1.5480000000000p-1, 0x1.a1b3071f75fdap-2}, {0x1.52a0000000000p-1, 0x1.a75a8a89c8c32p-2},
    {0x1.5100000000000p-1, 0x1.ac478d020506fp-2}, {0x1.4f40000000000p-1, 0x1.b19c6125a6f6bp-2},
    {0x1.4d80000000000p-1, 0x1.b6f859e8ef63ap-2}, {0x1.4be0000000000p-1, 0x1.bbf8c95e489bfp-2},
    {0x1.4a20000000000p-1, 0x1.c162bf5df23e5p-2}, {0x1.4880000000000p-1, 0x1.c6704e4016ff8p-2},
    {0x1.46e0000000000p-1, 0x1.cb844750b9995p-2}, {0x1.4540000000000p-1, 0x1.d09ebaee29dd8p-2},
    {0x1.43a0000000000p-1, 0x1.d5bfb9b5ae71fp-2}, {0x1.4200000000000p-1, 0x1.dae75484c9616p-2},
    {0x1.4080000000000p-1, 0x1.dfaf59de8c15dp-2}, {0x1.3ee0000000000p-1, 0x1.e4e3daeddb5f6p-2},
    {0x1.3d60000000000p-1, 0x1.e9b7e6610815ap-2}, {0x1.3be0000000000p-1, 0x1.ee91cce60d249p-2},
    {0x1.3a60000000000p-1, 0x1.f3719cc25c9b0p-2}, {0x1.38e0000000000p-1, 0x1.f857646fd4622p-2},
    {0x1.3760000000000p-1, 0x1.fd43329dc0365p-2}, {0x1.35e0000000000p-1, 0x1.011a8b18f0ed7p-1},
    {0x1.3460000000000p-1, 0x1.03968f24bfdb7p-1}, {0x1.3300000000000p-1, 0x1.05e04c1aa2c06p-1},
    {0x1.3180000000000p-1, 0x1.086248abc4f3bp-1}, {0x1.3020000000000p-1, 0x1.0ab18bf5823c3p-1},
    {0x1.2ec0000000000p-1, 0x1.0d037d237f464p-1}, {0x1.2d60000000000p-1, 0x1.0f5822744fca3p-1},
    {0x1.2be0000000000p-1, 0x1.11e62229bbf4ap-1}, {0x1.2aa0000000000p-1, 0x1.1409a2e6c81dap-1},
    {0x1.2940000000000p-1, 0x1.16668af4dd396p-1}, {0x1.27e0000000000p-1, 0x1.18c640ff75f06p-1},
    {0x1.2680000000000p-1, 0x1.1b28cbb6ec93fp-1}, {0x1.2540000000000p-1, 0x1.1d5650035a98bp-1},
    {0x1.23e0000000000p-1, 0x1.1fbe551db43c1p-1}, {0x1.22a0000000000p-1, 0x1.21f0dfc65ceecp-1},
    {0x1.2160000000000p-1, 0x1.2425d72bd3810p-1}, {0x1.2020000000000p-1, 0x1.265d40adef0b8p-1},
    {0x1.1ec0000000000p-1, 0x1.28d041990b0ebp-1}, {0x1.1d80000000000p-1, 0x1.2b0cdfbf7ad03p-1},
    {0x1.1c60000000000p-1, 0x1.2d1260ad99c76p-1}, {0x1.1b20000000000p-1, 0x1.2f53c9cc59422p-1},
    {0x1.19e0000000000p-1, 0x1.3197c0fa80e6ap-1}, {0x1.18a0000000000p-1, 0x1.33de4c086c40ap-1},
    {0x1.1780000000000p-1, 0x1.35eccf0ac61d0p-1}, {0x1.1640000000000p-1, 0x1.383850278cfd9p-1},
    {0x1.1520000000000p-1, 0x1.3a4b53f86cb2ep-1}, {0x1.1400000000000p-1, 0x1.3c6080c36bfb5p-1},
    {0x1.12c0000000000p-1, 0x1.3eb37978b85b5p-1}, {0x1.11a0000000000p-1, 0x1.40cd448ff6dd6p-1},
    {0x1.1080000000000p-1, 0x1.42e946de080bfp-1}, {0x1.0f60000000000p-1, 0x1.450785145cafep-1},
    {0x1.0e40000000000p-1, 0x1.472803f35eaaep-1}, {0x1.0d20000000000p-1, 0x1.494ac84ab0ed3p-1},
    {0x1.0c00000000000p-1, 0x1.4b6fd6f970c1fp-1}, {0x1.0b00000000000p-1, 0x1.4d59d43fdaba2p-1},
    {0x1.09e0000000000p-1, 0x1.4f8343f9cb679p-1}, {0x1.08c0000000000p-1, 0x1.51af0c774a2d0p-1},
    {0x1.07c0000000000p-1, 0x1.539f107e1d30ap-1}, {0x1.06a0000000000p-1, 0x1.55cf55c5a5438p-1},
    {0x1.05a0000000000p-1, 0x1.57c35f3490184p-1}, {0x1.04a0000000000p-1, 0x1.59b952dcd3e28p-1},
    {0x1.0380000000000p-1, 0x1.5bf053a48690ep-1}, {0x1.0280000000000p-1, 0x1.5dea65985a350p-1},
    {0x1.0180000000000p-1, 0x1.5fe66db228992p-1}, {0x1.0080000000000p-1, 0x1.61e46fda56467p-1},
};

// r = x - n ln2 / 128 with n = rint(128 x / ln2); |r| <= ln2 / 256
__device__ __forceinline__ double exp_reduce(double x, int& n) {
  const double t = fma(x, 0x1.71547652b82fep+7, 0x1.8p52);
  n = __double2loint(t);
  const double nd = t - 0x1.8p52;
  return fma(nd, -0x1.fdf473de6af28p-29, fma(nd, -0x1.62e4200000000p-8, x));
}
// 2^(n / 128) (1 + p)
__device__ __forceinline__ double exp_scale(int n, double p) {
  const double T = kExp2[n & 127];
  const double v = fma(T, p, T);
  return __hiloint2double(__double2hiint(v) + (n >> 7) * (1 << 20), __double2loint(v));
}
__device__ __forceinline__ bool exp_in_range(double x) { return (__double2hiint(x) & 0x7fffffff) < 0x4085e000; }  // |x| < 700

__device__ __forceinline__ double exp_fast(double x) {
  if (!exp_in_range(x)) return exp(x);
  int n;
  const double r = exp_reduce(x, n);
  const double q = fma(r, fma(r, fma(r, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5);
  return exp_scale(n, fma(r * r, q, r));
}

__device__ __forceinline__ void exp_pm_fast(double x, double& ep, double& em) {
  if (!exp_in_range(x)) {
    ep = exp(x);
    em = exp(-x);
    return;
  }
  int n;
  const double r = exp_reduce(x, n);
  const double r2 = r * r;
  const double ev = r2 * fma(r2, 1.0 / 24.0, 0.5);
  const double od = fma(r2 * r, fma(r2, 1.0 / 120.0, 1.0 / 6.0), r);
  ep = exp_scale(n, ev + od);
  em = exp_scale(-n, ev - od);
}

__device__ __forceinline__ bool positive_normal(double x) {
  const int h = __double2hiint(x);
  return h >= 0x00100000 && h < 0x7ff00000;
}

__device__ __forceinline__ double log_fast(double x) {   // positive_normal(x)
  const int h = __double2hiint(x);
  const double m = __hiloint2double((h & 0xfffff) | 0x3ff00000, __double2loint(x));
  const double2 cl = kLog[(h >> 13) & 127];
  const double e = __hiloint2double(0x43300000, ((h >> 20) - 1023) ^ 0x80000000) - 0x1.00000800p52;
  const double r = fma(m, cl.x, -1.0);                    // |r| < 0.00398
  const double q = fma(r, fma(r, fma(r, fma(r, -1.0 / 6.0, 0.2), -0.25), 1.0 / 3.0), -0.5);
  return fma(e, 0x1.62e42fefa39efp-1, cl.y) + fma(e, 0x1.abc9e3b39803fp-56, fma(r * r, q, r));
}

__device__ __forceinline__ double recip_fast(double x) {
  const int h = __double2hiint(x) & 0x7fffffff;
  if (h < 0x02000000 || h >= 0x7e000000) return 1.0 / x;   // keeps the seed and the steps normal
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}

}  // namespace dg
