// Pointwise fluxes and sources of the FP64 path (Eq. fluxSWNondimensional, Eq. LDG2) in the form with the
// fewest FP64 instructions. S is double or the dual number DualT<double>.
//
// The generic expressions of dg_internal.cuh scale every velocity and temperature gradient by
// 1/sqrt(rho) and form the stress from the scaled ones. Here the unscaled w = grad u_m - u_m grad(varrho)/2
// is kept: with s = 1/sqrt(rho), e = w + w^T - (2/3) tr(w) I,
//   viscous flux      tau = (c_mu mu s^2) e          (= c_mu mu s eps)
//   heat flux         h = (c_k kappa s^2 / c_v) w_T
//   div v = s tr(w),  sqrt(rho) T div v = T tr(w),   sqrt(rho) omega x v = omega x u
//   dissipation       c_d mu s eps : grad v / c_v = (c_d / (c_mu c_v)) s (tau : w)
// tau is symmetric, so six products serve the flux, the momentum source and the dissipation. A value and
// its tangent take about 270 FP64 instructions per volume point and 420 per face point besides the
// reference-space contraction (640 and 960 before, with CUDA's exp, log and divisions).
#pragma once

#include "dg_euvac64.cuh"
#include "dg_internal.cuh"
#include "dg_math64.cuh"

namespace dg {

using D64 = DualT<double>;
__device__ __forceinline__ double s_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ D64 s_fma(D64 a, D64 b, D64 c) {
  return {fma(a.v, b.v, c.v), fma(a.v, b.d, fma(a.d, b.v, c.d))};
}
__device__ __forceinline__ D64 s_fma(double a, D64 b, D64 c) { return {fma(a, b.v, c.v), fma(a, b.d, c.d)}; }

__device__ __forceinline__ double val64(double x) { return x; }
__device__ __forceinline__ double val64(D64 x) { return x.v; }
// f(k) of value f and derivative df
__device__ __forceinline__ double tangent64(double f, double, double) { return f; }
__device__ __forceinline__ D64 tangent64(double f, double df, D64 k) { return {f, df * k.d}; }

// s = e^{-varrho/2}, sr = e^{varrho/2}
__device__ __forceinline__ void s_rho(double u0, double& s, double& sr) { exp_pm_fast(0.5 * u0, sr, s); }
__device__ __forceinline__ void s_rho(D64 u0, D64& s, D64& sr) {
  const double hd = 0.5 * u0.d;
  exp_pm_fast(0.5 * u0.v, sr.v, s.v);
  s.d = -s.v * hd;
  sr.d = sr.v * hd;
}
__device__ __forceinline__ double s_isr(double u0) { return exp_fast(-0.5 * u0); }
__device__ __forceinline__ D64 s_isr(D64 u0) {
  const double s = exp_fast(-0.5 * u0.v);
  return {s, s * (-0.5 * u0.d)};
}

// T^a with T = u4 e^{-varrho/2}: exp(a (log u4 - varrho/2)); dl is d(log T) of the tangent
__device__ __forceinline__ double t_power(double a, double u0, double u4, double dl) {
  (void)dl;
  return power_fast(a, u4, u0);
}
__device__ __forceinline__ D64 t_power(double a, D64 u0, D64 u4, double dl) {
  const double p = t_power(a, u0.v, u4.v, 0.0);
  return {p, (a * p) * dl};
}
__device__ __forceinline__ double t_dlog(double, double) { return 0.0; }
__device__ __forceinline__ double t_dlog(D64 u0, D64 u4) { return fma(-0.5, u0.d, u4.d * recip_fast(u4.v)); }

// viscosity over c_mu (mu) and conductivity (kappa); the law T^visc_exp has kappa = mu
template <typename S>
__device__ __forceinline__ void transport64(const PhysT<double>& P, const S& u0, const S& u4, const S& s,
                                            const Mix<double>& mx, S& mu, S& kappa) {
  if (P.comp) {
    const S T = u4 * s;
    const S rho = s_inv(s * s);
    mu = s_sqrt(T * (1.0 / mx.cv)) + P.eddy_nu * rho;
    kappa = mx.kfac * t_power(0.69, u0, u4, t_dlog(u0, u4)) + (P.eddy_alpha * mx.cv) * rho;
  } else {
    mu = P.visc_exp != 0.0 ? t_power(P.visc_exp, u0, u4, t_dlog(u0, u4)) : s_const<S>(1.0);
    kappa = mu;
  }
}

// the unscaled gradients and the viscous coefficients of one point
template <typename S>
struct Grad64 {
  S w[3][3];          // w[d][m] = d u_m / d x_d - u_m (d varrho / d x_d) / 2
  S wT[3], tr;
  S e[6];             // xx, yy, zz, xy, xz, yz
};
template <typename S>
__device__ __forceinline__ void gradients64(const S u[5], const S q[3][5], Grad64<S>& g) {
  S h[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) h[m] = -0.5 * u[1 + m];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
#pragma unroll
    for (int m = 0; m < 3; ++m) g.w[d][m] = s_fma(h[m], q[d][0], q[d][1 + m]);
    g.wT[d] = s_fma(h[3], q[d][0], q[d][4]);
  }
  g.tr = g.w[0][0] + g.w[1][1] + g.w[2][2];
  const S third = (-2.0 / 3.0) * g.tr;
#pragma unroll
  for (int m = 0; m < 3; ++m) g.e[m] = s_fma(2.0, g.w[m][m], third);
  g.e[3] = g.w[0][1] + g.w[1][0];
  g.e[4] = g.w[0][2] + g.w[2][0];
  g.e[5] = g.w[1][2] + g.w[2][1];
}
template <typename S>
__device__ __forceinline__ void viscous64(const PhysT<double>& P, const S& mu, const S& kappa, const S& s, double cv,
                                          S& K, S& K2) {
  const S s2 = s * s;
  K = (P.c_mu * mu) * s2;
  K2 = P.comp ? ((P.c_k / cv) * kappa) * s2 : (P.c_k / (cv * P.c_mu)) * K;
}

// F(u, q) . n with the viscous terms; K, K2 the viscous coefficients
template <typename S>
__device__ __forceinline__ void flux_n64(const PhysT<double>& P, const S u[5], const S q[3][5], const double n[3],
                                         double pc, const S& s, const S& K, const S& K2, S out[5]) {
  Grad64<S> g;
  gradients64(u, q, g);
  const S vn = s * s_fma(n[0], u[1], s_fma(n[1], u[2], n[2] * u[3]));
  const S en[3] = {s_fma(n[0], g.e[0], s_fma(n[1], g.e[3], n[2] * g.e[4])),
                   s_fma(n[0], g.e[3], s_fma(n[1], g.e[1], n[2] * g.e[5])),
                   s_fma(n[0], g.e[4], s_fma(n[1], g.e[5], n[2] * g.e[2]))};
  out[0] = u[0] * vn;
  const S nK = -1.0 * K;
#pragma unroll
  for (int m = 0; m < 3; ++m) out[1 + m] = s_fma(u[1 + m], vn, s_fma(nK, en[m], (pc * n[m]) * u[4]));
  out[4] = s_fma(u[4], vn, -1.0 * (K2 * s_fma(n[0], g.wT[0], s_fma(n[1], g.wT[1], n[2] * g.wT[2]))));
}
// without them (outflow)
template <typename S>
__device__ __forceinline__ void flux_n64_inviscid(const S u[5], const double n[3], double pc, const S& s, S out[5]) {
  const S vn = s * s_fma(n[0], u[1], s_fma(n[1], u[2], n[2] * u[3]));
  out[0] = u[0] * vn;
#pragma unroll
  for (int m = 0; m < 3; ++m) out[1 + m] = s_fma(u[1 + m], vn, (pc * n[m]) * u[4]);
  out[4] = u[4] * vn;
}
// the part of the flux's tangent that a tangent dq of the gradient alone makes (linear in dq)
__device__ __forceinline__ void flux_n64_dq(const double u[5], const double dq[3][5], const double n[3], double K,
                                            double K2, double out[5]) {
  Grad64<double> g;
  gradients64(u, dq, g);
  const double nK = -K;
  out[0] = 0.0;
  out[1] = nK * fma(n[0], g.e[0], fma(n[1], g.e[3], n[2] * g.e[4]));
  out[2] = nK * fma(n[0], g.e[3], fma(n[1], g.e[1], n[2] * g.e[5]));
  out[3] = nK * fma(n[0], g.e[4], fma(n[1], g.e[5], n[2] * g.e[2]));
  out[4] = -K2 * fma(n[0], g.wT[0], fma(n[1], g.wT[1], n[2] * g.wT[2]));
}

// s, viscous coefficients of a state
template <typename S>
__device__ __forceinline__ void state64(const PhysT<double>& P, const S u[5], const Mix<double>& mx, S& s, S& K, S& K2) {
  s = s_isr(u[0]);
  S mu, kappa;
  transport64(P, u[0], u[4], s, mx, mu, kappa);
  viscous64(P, mu, kappa, s, P.comp ? mx.cv : P.cv, K, K2);
}

// stabilisation: sigma = lambda0 on varrho, sm on the momentum, se on the energy (at the trace uh)
template <typename S>
__device__ __forceinline__ void sigma64(const PhysT<double>& P, const S& uh0, const S& uh4, const Mix<double>& mx, S& sm,
                                        S& se) {
  const S s = s_isr(uh0);
  S mu, kappa;
  transport64(P, uh0, uh4, s, mx, mu, kappa);
  const S x = (P.c_mu * mu) * s;
  sm = P.lam + x;
  se = P.comp ? P.lam + ((P.c_k / mx.cv) * kappa) * s : P.lam + (P.c_k / (P.cv * P.c_mu)) * x;
}

// the Sun at the time of the call (host): unit direction for EUVAC, (cos, sin) of the rotation for the
// Gaussian, and the band tables
struct Sun64 {
  double d[3];
  const EuvFx* bands;
};

// EUVAC / Gaussian heating over c_v sqrt(rho), added to the energy source
template <typename S>
__device__ __forceinline__ S heating64(const PhysT<double>& P, const Sun64& sun, const S& s, const S& sr, const S& T,
                                       double cvp, const double* xg, const double mg[8]) {
  const double r2 = xg[0] * xg[0] + xg[1] * xg[1] + xg[2] * xg[2];
  const double r = sqrt(r2), ir = recip_fast(r), icv = recip_fast(cvp);
  double cchi = (xg[0] * sun.d[0] + xg[1] * sun.d[1] + xg[2] * sun.d[2]) * ir;
  cchi = fmin(1.0, fmax(-1.0, cchi));
  if (P.euv == DG_EUV_GAUSS) {
    const double chi = acos(cchi);
    const double dz = (r - P.euv_r_peak) * P.euv_inv_w;
    const double Qh = P.euv_amp * exp_fast(fma(-chi * chi, P.euv_inv2s2, -0.6931471805599453 * dz * dz));
    return (Qh * icv) * s;
  }
  const double schi = sqrt(fmax(0.0, 1.0 - cchi * cchi));
  if (!(cchi > 0.0 || schi * r > P.g_r0)) return s_zero<S>();   // in the Earth's shadow
  const S er = sr * sr;                             // e^varrho
  const double minv = P.comp ? cvp : P.inv_m;       // 1/m*
  const S Hs = T * (r2 * minv / (P.g_r0 * P.g_r0));   // H* = T* r*^2 / (m* g_r0^2)
  const S rt = r * s_inv(Hs);                       // r~ = |r| / H
  const S hr = s_sqrt(0.5 * rt);
  const S ex = s_erfcx(hr * fabs(cchi));
  const S base = 1.7724538509055160273 * hr;        // sqrt(pi r~ / 2)
  S ch;
  if (cchi > 0.0) ch = base * ex;
  else ch = base * (2.0 * s_exp(rt * (1.0 - schi)) - ex);
  // species weights w_s = chi_s / m_s* (O, N2, O2, He), or 1/m* on oxygen alone
  const S k = (P.euvac_cc * er) * Hs * ch;          // tau_j = Phi_j k
  const double kv = val64(k);
  double S0, S1;
  if (P.comp) {
    const double ws[4] = {1.0 - mg[5] - mg[6] - mg[7], mg[5] * (16.0 / 28.0), mg[6] * (16.0 / 32.0), mg[7] * (16.0 / 4.0)};
    euvac_sums<4>(sun.bands, ws, kv, S0, S1);
  } else {
    const double ws[4] = {1.0, 0.0, 0.0, 0.0};
    euvac_sums<1>(sun.bands, ws, P.inv_m * kv, S0, S1);
    S0 *= P.inv_m;
    S1 *= P.inv_m * P.inv_m;
  }
  return (er * tangent64(S0, -S1, k)) * icv * s;
}

// physical fluxes F[12]: momentum xx, yy, zz, xy, xz, yz (symmetric), varrho x, y, z, energy x, y, z; and
// the sources, weighted with the Jacobian determinant
template <typename S>
__device__ __forceinline__ void volume64(const PhysT<double>& P, const S u[5], const S q[3][5], double det,
                                         const double acc[3], const double* xg, const Sun64& sun, const double mg[8], S F[12],
                                         S src[5]) {
  const Mix<double> mx{P.comp ? mg[0] : P.cv, P.comp ? mg[4] : 1.0};
  const double cvp = mx.cv;
  const double pc = P.comp ? cvp * P.inv_gamma : P.p_coef;   // 1/(gamma m*)
  S s, sr, mu, kappa, K, K2;
  s_rho(u[0], s, sr);
  transport64(P, u[0], u[4], s, mx, mu, kappa);
  viscous64(P, mu, kappa, s, cvp, K, K2);
  Grad64<S> g;
  gradients64(u, q, g);
  S tau[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) tau[k] = K * g.e[k];
  const S pr = pc * u[4];
  // P_md = p delta - tau
  const S Pm[6] = {pr - tau[0], pr - tau[1], pr - tau[2], -tau[3], -tau[4], -tau[5]};
  const S hT[3] = {-1.0 * (K2 * g.wT[0]), -1.0 * (K2 * g.wT[1]), -1.0 * (K2 * g.wT[2])};
  S hq[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) hq[d] = -0.5 * q[d][0];
  // sources
  const S divv = s * g.tr;
  src[0] = det * s_fma(u[0], divv, -divv);
  const double* om = P.omega;
  const S rot[3] = {om[1] * u[3] - om[2] * u[2], om[2] * u[1] - om[0] * u[3], om[0] * u[2] - om[1] * u[1]};
  constexpr int ix[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  const S hdiv = 0.5 * divv;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    S x = s_fma(acc[m], sr, -P.cor * rot[m]);
    x = s_fma(hdiv, u[1 + m], x);
#pragma unroll
    for (int d = 0; d < 3; ++d) x = s_fma(Pm[ix[m][d]], hq[d], x);
    src[1 + m] = det * x;
  }
  S dis = tau[0] * g.w[0][0];
  dis = s_fma(tau[1], g.w[1][1], dis);
  dis = s_fma(tau[2], g.w[2][2], dis);
#pragma unroll
  for (int k = 3; k < 6; ++k) dis = s_fma(tau[k], g.e[k], dis);
  const S T = u[4] * s;
  S x = ((1.5 - P.gamma) * T) * g.tr;
  x = s_fma((P.c_d / (cvp * P.c_mu)) * s, dis, x);
#pragma unroll
  for (int d = 0; d < 3; ++d) x = s_fma(hT[d], hq[d], x);
  // fluxes
  const S v[3] = {u[1] * s, u[2] * s, u[3] * s};
  F[0] = s_fma(u[1], v[0], Pm[0]);
  F[1] = s_fma(u[2], v[1], Pm[1]);
  F[2] = s_fma(u[3], v[2], Pm[2]);
  F[3] = s_fma(u[1], v[1], Pm[3]);
  F[4] = s_fma(u[1], v[2], Pm[4]);
  F[5] = s_fma(u[2], v[2], Pm[5]);
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    F[6 + d] = u[0] * v[d];
    F[9 + d] = s_fma(u[4], v[d], hT[d]);
  }
  if (P.comp) {
    // -(1/c_v) (sqrt(rho) T v - c_kappa kappa / (sqrt(rho) c_v) grad T) . grad c_v
    const double icv = -1.0 / cvp;
#pragma unroll
    for (int d = 0; d < 3; ++d) x = s_fma(icv * mg[1 + d], F[9 + d], x);
  }
  if (P.euv) x = x + heating64(P, sun, s, sr, T, cvp, xg, mg);
  src[4] = det * x;
}

}  // namespace dg
