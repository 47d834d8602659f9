// Block fixed-point arithmetic for the FP64 basis contractions, on the integer pipe.
//
// GB300 issues 2 FP64 thread-operations per SM and cycle and 64 integer multiply-adds (32 x 32 + 64
// bits), 32 for one; eight mad.wide issued beside each DFMA cost no time at all (measured: 8 DFMA per
// iteration 1.10 ms, with 64 mad.wide added 1.12 ms). The contractions of the FP64 path have constant
// coefficients and one element of data, so they run in fixed point with one exponent per element and
// variable:
//   data         X = round(x 2^S), |X| <= 2^58, S from the largest magnitude in the element, held as
//                X = h1 2^LH + h0 with 0 <= h0 < 2^LH (one int2, the 8 bytes of the double it stands for)
//   coefficient  A = round(a 2^t) = a1 2^LA + a0 with -2^(LA-1) <= a0 < 2^(LA-1), LA + LH = 57
//   sum          H += a1 h1,  M += a1 h0,  L += a0 h1   (three mad.wide per term; a0 h0 is left out)
//   result       R = H + (M >> LH) + (L >> LA) = sum(A X) 2^-57 up to about one unit
// The splits put as many bits as the sums allow into a1 and h1, so that the omitted a0 h0 stays below
// the result's unit: LA = 29, LH = 28 for the weak derivative with lifting; LA = 27, LH = 30 for
// interpolation and face traces, whose data grow by the passes. Data are rounded at 2^-58 of the largest
// magnitude in the element and sums do not round, so the result is closer to exact than FP64 FMA chains
// (2^-53 of every partial sum). Exponents outside the range checked by the kernels (zero fields are fine;
// Inf, NaN and magnitudes whose products could leave the normal FP64 range are not) take the FP64 path in
// the same kernel.
//
// Quadrature weights would make the data of one element differ by up to 14 (5 points), so the FP64
// kernels hold cofactors and normals without them and the weights are folded into the coefficients:
// Dh[k][i] = D[k][i] w_k / w_i, eh[i] = e[i] / w_i (both sides divided by the weight of the result's
// point), Bt[q][a] = B[q][a] w_q.
// Overflow: with the column sums of the operators for 2 to 5 points (weak derivative with lifting: 10.4,
// 19.9, 32.0, 47.0; |B| rows 1.39, |Bt| columns 1.34; end-point rows 3.33) every accumulator stays below
// 2^63; the exponents t and the data widths are chosen for that.
#pragma once

#include <cuda_runtime.h>

namespace dg {

constexpr int FX_T_B = 57;     // |B|, |Bt| <= 1
constexpr int FX_T_D = 56;     // |Dh| <= 5.07, |eh| <= 6.55, sums with lifting <= 47.0
constexpr int FX_T_E = 57;     // |eL|, |eR| <= 1.56

struct fx { int hi, lo; };     // X = hi 2^LH + lo

template <int LH>
__device__ __forceinline__ fx fx_split(long long X) { return {(int)(X >> LH), (int)X & ((1 << LH) - 1)}; }
template <int LH>
__device__ __forceinline__ long long fx_join(fx x) { return ((long long)x.hi << LH) + x.lo; }

// round(x 2^S) with S = BITS + 1022 - emax, for |x| < 2^(emax - 1022)
template <int BITS>
__device__ __forceinline__ long long fx_from(double x, int emax) {
  const int hi = __double2hiint(x);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  const int d = min(emax - e, 63);
  const long long X = (long long)((((m << (BITS - 52)) >> d) + 1) >> 1);
  return hi < 0 ? -X : X;
}

// R 2^sh as a double: one conversion on the FP64 pipe and an exponent add
__device__ __forceinline__ double fx_to_double(long long R, int sh) {
  const double d = (double)R;
  const int hi = __double2hiint(d);
  return __hiloint2double(R ? hi + (sh << 20) : hi, __double2loint(d));
}

struct fxacc { long long H, M, L; };
template <int LH>
__device__ __forceinline__ fxacc fx_zero() { return {0, 1LL << (LH - 1), 0}; }
__device__ __forceinline__ void fx_mac(fxacc& s, fx a, fx x) {
#ifdef __CUDA_ARCH__
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.H) : "r"(a.hi), "r"(x.hi));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.M) : "r"(a.hi), "r"(x.lo));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(s.L) : "r"(a.lo), "r"(x.hi));
#else
  s.H += (long long)a.hi * x.hi;
  s.M += (long long)a.hi * x.lo;
  s.L += (long long)a.lo * x.hi;
#endif
}
template <int LH>
__device__ __forceinline__ long long fx_sum(const fxacc& s) { return s.H + (s.M >> LH) + (s.L >> (57 - LH)); }
// product of two data values times 2^-57: x split at 57 - LH, y at LH
template <int LH>
__device__ __forceinline__ long long fx_mul(fx x, fx y) {
  fxacc s = fx_zero<LH>();
  fx_mac(s, x, y);
  return fx_sum<LH>(s);
}

// biased exponent bound of a maximum of magnitude words (see fx_mag), and whether it is usable
__device__ __forceinline__ int fx_mag(double x) {      // high word of |x|; 1 for nonzero below 2^-1042
  const int h = __double2hiint(x) & 0x7fffffff;
  return (h == 0 && __double2loint(x) != 0) ? 1 : h;
}
__device__ __forceinline__ int fx_exp(int mag) { return mag == 0 ? 1023 : mag >> 20; }
__device__ __forceinline__ bool fx_ok(int mag) { return mag == 0 || ((mag >> 20) >= 200 && (mag >> 20) <= 1846); }

// host: coefficient with exponent t, split at LA
inline int2 fx_coef(long double a, int t, int LA) {
  const long long A = (long long)__builtin_llrintl(__builtin_ldexpl(a, t));
  const long long a1 = (A + (1LL << (LA - 1))) >> LA;
  return make_int2((int)a1, (int)(A - (a1 << LA)));
}

}  // namespace dg
