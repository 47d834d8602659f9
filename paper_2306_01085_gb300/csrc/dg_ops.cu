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
// more than the rounding of the data.
using ld = long double;

// Legendre P_n(x) and its derivative by the three-term recurrence
void legendre(int n, ld x, ld* p, ld* dp) {
  ld p0 = 1.0L, p1 = x;
  if (n == 0) { *p = 1.0L; *dp = 0.0L; return; }
  for (int k = 2; k <= n; ++k) {
    ld p2 = ((2.0L * k - 1.0L) * x * p1 - (k - 1.0L) * p0) / k;
    p0 = p1;
    p1 = p2;
  }
  *p = p1;
  *dp = (std::fabs(x) < 1.0L) ? n * (p0 - x * p1) / (1.0L - x * x) : 0.5L * n * (n + 1) * std::pow(x, n + 1);
}

// Gauss-Legendre: roots of P_n by Newton from Chebyshev-like guesses, weights 2/((1-x^2) P_n'^2)
void gauss_rule(int n, ld* x, ld* w) {
  for (int i = 0; i < n; ++i) {
    ld z = -std::cos((ld)M_PI * (i + 0.75L) / (n + 0.5L));
    if (2 * i + 1 == n) z = 0.0L;
    for (int it = 0; it < 100; ++it) {
      ld p, dp;
      legendre(n, z, &p, &dp);
      ld dz = p / dp;
      z -= dz;
      if (std::fabs(dz) < 1e-19L) break;
    }
    ld p, dp;
    legendre(n, z, &p, &dp);
    x[i] = z;
    w[i] = 2.0L / ((1.0L - z * z) * dp * dp);
  }
}

// GLL nodes: -1, roots of P'_{n-1}, +1. Newton on q(x) = (1 - x^2) P'_{n-1}(x), whose
// derivative is -(n-1) n P_{n-1}(x) (Legendre's equation).
void gll_nodes(int n, ld* x) {
  int N = n - 1;
  x[0] = -1.0L;
  x[N] = 1.0L;
  for (int i = 1; i < N; ++i) {
    ld z = -std::cos((ld)M_PI * i / N);
    if (2 * i == N) z = 0.0L;
    for (int it = 0; it < 100; ++it) {
      ld p, dp;
      legendre(N, z, &p, &dp);
      ld qv = (1.0L - z * z) * dp;
      ld dq = -ld(N) * (N + 1) * p;
      ld dz = qv / dq;
      z -= dz;
      if (std::fabs(dz) < 1e-19L) break;
    }
    x[i] = z;
  }
}

// barycentric weights of a node set
void bary(int n, const ld* x, ld* lam) {
  for (int k = 0; k < n; ++k) {
    ld prod = 1.0L;
    for (int m = 0; m < n; ++m)
      if (m != k) prod *= (x[k] - x[m]);
    lam[k] = 1.0L / prod;
  }
}

// Lagrange basis of node set x evaluated at point t: out[k] = l_k(t) (product form)
void lagrange_at(int n, const ld* x, ld t, ld* out) {
  for (int k = 0; k < n; ++k) {
    ld v = 1.0L;
    for (int m = 0; m < n; ++m)
      if (m != k) v *= (t - x[m]) / (x[k] - x[m]);
    out[k] = v;
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
  // derivative matrix on the Gauss points: D[q][k] = lam_k / lam_q / (eta_q - eta_k), q != k;
  // the diagonal makes every row sum to zero (derivative of a constant)
  ld lam[MAXN];
  bary(n, o->eta, lam);
  for (int q = 0; q < n; ++q) {
    ld diag = 0.0L;
    for (int k = 0; k < n; ++k) {
      if (k == q) continue;
      ld v = lam[k] / lam[q] / (o->eta[q] - o->eta[k]);
      o->D[q * n + k] = v;
      diag -= v;
    }
    o->D[q * n + q] = diag;
  }
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
