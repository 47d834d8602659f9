// FP64 exponentials, powers and reciprocals of the pointwise physics with few FP64 instructions.
//
// GB300 has 2 FP64 lanes per SM, so an FP64 instruction costs a warp 64 issue cycles of its scheduler
// while table look-ups and integer instructions are nearly free beside it.
//   exp_fast, exp_pm_fast, power_fast   fixed point (dg_exp_fx.cuh), no FP64 instruction; outside its ranges
//                                       (and for Inf, NaN) CUDA's exp and log
//   recip_fast     4 FP64 instructions: two Newton-Raphson steps y + y (1 - x y) from the hardware's seed, which is good
//                  to 2^-20; the second leaves 2^-80 before its rounding, so the error is below 0.5 + 2^-20 ulp
//                  (a division is correctly rounded); outside 2^-991 <= |x| < 2^993 the division itself
#pragma once

#include <cuda_runtime.h>

#include "dg_exp_fx.cuh"

namespace dg {

static __device__ __noinline__ double exp_slow(double x) { return exp(x); }

__device__ __forceinline__ double exp_fast(double x) { return fx_exp_range(x) ? fx_exp(x) : exp_slow(x); }

__device__ __forceinline__ void exp_pm_fast(double x, double& ep, double& em) {
  if (fx_exp_range(x)) {
    fx_exp_pm(x, ep, em);
  } else {
    ep = exp_slow(x);
    em = exp_slow(-x);
  }
}

__device__ __forceinline__ bool positive_normal(double x) {
  const int h = __double2hiint(x);
  return h >= 0x00100000 && h < 0x7ff00000;
}

// u^a e^(-a v / 2)
static __device__ __noinline__ double power_slow(double a, double u, double v) {
  if (!positive_normal(u)) return exp(a * log(u * exp(-0.5 * v)));
  return exp(a * fma(-0.5, v, log(u)));
}
__device__ __forceinline__ double power_fast(double a, double u, double v) {
  return fx_power_range(a, u, v) ? fx_power(a, u, v) : power_slow(a, u, v);
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
