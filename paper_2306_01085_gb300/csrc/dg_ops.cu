// 1D quadrature and Lagrange operators of the tensor-product DG basis (host code).
//
// Sec. 3.1: the element spaces hold polynomials of degree k = n - 1. The library represents them by
// the Lagrange basis on n Gauss-Lobatto-Legendre (GLL) nodes (the nodal layout of the ABI) and
// integrates with the n-point Gauss-Legendre rule. Internally the kernels work with values at the
// Gauss points (the map between the two is the invertible tensor matrix B x B x B).
#include <cmath>
#include <cstring>

#include "dg_internal.cuh"

namespace dg {

namespace {

// The operators are formed in extended precision and rounded once: their errors act on every element
// alike (a row of B that sums to 1 + 1e-16 turns a large constant into a gradient), so they are worth
// more than the rounding of the data. The same code in double serves the geometry (build_ops_geo).
using ld = long double;

// Legendre P_n(x) and its derivative by the three-term recurrence
template <typename T>
void legendre(int n, T x, T* p, T* dp) {
  T p0 = T(1.0), p1 = x;
  if (n == 0) { *p = T(1.0); *dp = T(0.0); return; }
  for (int k = 2; k <= n; ++k) {
    T p2 = ((T(2.0) * k - T(1.0)) * x * p1 - (k - T(1.0)) * p0) / k;
    p0 = p1;
    p1 = p2;
  }
  *p = p1;
  *dp = (std::fabs(x) < T(1.0)) ? n * (p0 - x * p1) / (T(1.0) - x * x) : T(0.5) * n * (n + 1) * std::pow(x, n + 1);
}

// Gauss-Legendre: roots of P_n by Newton from Chebyshev-like guesses, weights 2/((1-x^2) P_n'^2)
template <typename T>
void gauss_rule(int n, T* x, T* w) {
  for (int i = 0; i < n; ++i) {
    T z = -std::cos(T(M_PI) * (i + T(0.75)) / (n + T(0.5)));
    if (sizeof(T) > sizeof(double) && 2 * i + 1 == n) z = T(0.0);
    const T tol = sizeof(T) > sizeof(double) ? T(1e-19L) : T(1e-16);
    for (int it = 0; it < 100; ++it) {
      T p, dp;
      legendre(n, z, &p, &dp);
      T dz = p / dp;
      z -= dz;
      if (std::fabs(dz) < tol) break;
    }
    T p, dp;
    legendre(n, z, &p, &dp);
    x[i] = z;
    w[i] = T(2.0) / ((T(1.0) - z * z) * dp * dp);
  }
}

// GLL nodes: -1, roots of P'_{n-1}, +1. Newton on q(x) = (1 - x^2) P'_{n-1}(x), whose
// derivative is -(n-1) n P_{n-1}(x) (Legendre's equation).
template <typename T>
void gll_nodes(int n, T* x) {
  int N = n - 1;
  x[0] = -T(1.0);
  x[N] = T(1.0);
  for (int i = 1; i < N; ++i) {
    T z = -std::cos(T(M_PI) * i / N);
    if (sizeof(T) > sizeof(double) && 2 * i == N) z = T(0.0);
    const T tol = sizeof(T) > sizeof(double) ? T(1e-19L) : T(1e-16);
    for (int it = 0; it < 100; ++it) {
      T p, dp;
      legendre(N, z, &p, &dp);
      T qv = (T(1.0) - z * z) * dp;
      T dq = -T(N) * (N + 1) * p;
      T dz = qv / dq;
      z -= dz;
      if (std::fabs(dz) < tol) break;
    }
    x[i] = z;
  }
}

// barycentric weights of a node set
template <typename T>
void bary(int n, const T* x, T* lam) {
  for (int k = 0; k < n; ++k) {
    T prod = T(1.0);
    for (int m = 0; m < n; ++m)
      if (m != k) prod *= (x[k] - x[m]);
    lam[k] = T(1.0) / prod;
  }
}

// Lagrange basis of node set x evaluated at point t: out[k] = l_k(t) (product form)
template <typename T>
void lagrange_at(int n, const T* x, T t, T* out) {
  for (int k = 0; k < n; ++k) {
    T v = T(1.0);
    for (int m = 0; m < n; ++m)
      if (m != k) v *= (t - x[m]) / (x[k] - x[m]);
    out[k] = v;
  }
}

// derivative matrix on the Gauss points: D[q][k] = lam_k / lam_q / (eta_q - eta_k), q != k;
// the diagonal makes every row sum to zero (derivative of a constant)
template <typename T>
void derivative(int n, const T* eta, T* D) {
  T lam[MAXN];
  bary(n, eta, lam);
  for (int q = 0; q < n; ++q) {
    T diag = T(0.0);
    for (int k = 0; k < n; ++k) {
      if (k == q) continue;
      T v = lam[k] / lam[q] / (eta[q] - eta[k]);
      D[q * n + k] = v;
      diag -= v;
    }
    D[q * n + q] = diag;
  }
}

}  // namespace

void build_ops_ld(int n, OpsLd* o) {
  gauss_rule(n, o->eta, o->w);
  gll_nodes(n, o->xi);
  for (int q = 0; q < n; ++q) lagrange_at(n, o->xi, o->eta[q], o->B + q * n);
  for (int a = 0; a < n; ++a) lagrange_at(n, o->eta, o->xi[a], o->Binv + a * n);
  lagrange_at(n, o->eta, -1.0L, o->e[0]);
  lagrange_at(n, o->eta, 1.0L, o->e[1]);
  derivative(n, o->eta, o->D);
}

void build_ops_geo(int n, Ops* o) {
  std::memset(o, 0, sizeof(Ops));
  gauss_rule(n, o->eta, o->w);
  gll_nodes(n, o->xi);
  for (int q = 0; q < n; ++q) lagrange_at(n, o->xi, o->eta[q], o->B + q * n);
  for (int a = 0; a < n; ++a) lagrange_at(n, o->eta, o->xi[a], o->Binv + a * n);
  lagrange_at(n, o->eta, -1.0, o->eL);
  lagrange_at(n, o->eta, 1.0, o->eR);
  derivative(n, o->eta, o->D);
}

void build_ops(int n, Ops* o) {
  std::memset(o, 0, sizeof(Ops));
  OpsLd L;
  build_ops_ld(n, &L);
  for (int k = 0; k < n; ++k) {
    o->eta[k] = (double)L.eta[k];
    o->w[k] = (double)L.w[k];
    o->iw[k] = (double)(1.0L / L.w[k]);
    o->xi[k] = (double)L.xi[k];
    o->eL[k] = (double)L.e[0][k];
    o->eR[k] = (double)L.e[1][k];
  }
  for (int q = 0; q < n; ++q)
    for (int k = 0; k < n; ++k) {
      const int i = q * n + k;
      const ld Dh = L.D[i] * L.w[q] / L.w[k], Bt = L.B[i] * L.w[q];
      o->B[i] = (double)L.B[i];
      o->Binv[i] = (double)L.Binv[i];
      o->D[i] = (double)L.D[i];
      o->Dh[i] = (double)Dh;
      o->Bt[i] = (double)Bt;
      o->xB[i] = fx_coef(L.B[i], FX_T_B, 27);
      o->xBt[i] = fx_coef(Bt, FX_T_B, 27);
      o->xBinv[i] = fx_coef(L.Binv[i], FX_T_B, 27);
      o->xDn[i] = fx_coef(-Dh, FX_T_D, 29);
    }
  for (int side = 0; side < 2; ++side)
    for (int k = 0; k < n; ++k) {
      const ld eh = L.e[side][k] / L.w[k];
      o->eh[side][k] = (double)eh;
      o->xlift[side][k] = fx_coef(eh, FX_T_D, 29);
      o->xend[side][k] = fx_coef(L.e[side][k], FX_T_E, 27);
    }
}

}  // namespace dg
