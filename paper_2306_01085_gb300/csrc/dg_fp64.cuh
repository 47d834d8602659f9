// FP64 kernels of the residual and its tangent whose basis contractions run in block fixed point
// (dg_fx.cuh); pointwise physics stays FP64. Included by dg_kernels.cuh, which holds the operators'
// formulation, the FP32 kernels and the pointwise functions.
//
// Layout of the work: one group of T threads per element and plane (value or tangent), T the number of
// Gauss points rounded up to 8 (2 points per direction), 32, 64 or 128, thread = Gauss point. Groups of
// up to a warp synchronise with __syncwarp and share a CTA with others; larger ones are a CTA of their
// own. A value and its tangent never mix in interpolation and gradient, so a tangent computed alone is
// bit for bit the tangent computed beside its value.
// Every contraction has an FP64 twin (the !FX branches) for elements whose magnitudes the fixed-point
// range check refuses (Inf, NaN, near the ends of the FP64 range): same formulas, FP64 FMA chains.
#pragma once

namespace dg {

template <int N>
struct Grp {
  static constexpr int NP = N * N * N, NF = N * N;
  static constexpr int T = N == 2 ? 8 : (NP + 31) / 32 * 32;
  static constexpr int W = T / 32;            // warps of a group (0: several groups per warp)
  static constexpr int NI = (6 * NF + T - 1) / T;   // face points per thread
};

template <int N>
__device__ __forceinline__ void grp_sync() {
  if constexpr (Grp<N>::T <= 32) __syncwarp();
  else __syncthreads();
}

// largest of each of K words over the group's threads; red: shared [W][K] of the group (W > 1 only),
// reusable after the next grp_sync
template <int N, int K>
__device__ __forceinline__ void grp_max(int (&v)[K], int* red) {
  constexpr int T = Grp<N>::T, W = Grp<N>::W;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if constexpr (T < 32) {
#pragma unroll
      for (int off = T / 2; off > 0; off >>= 1) v[k] = max(v[k], __shfl_xor_sync(0xffffffffu, v[k], off));
    } else {
      v[k] = __reduce_max_sync(0xffffffffu, v[k]);
    }
  }
  if constexpr (W > 1) {
    const int warp = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) red[warp * K + k] = v[k];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int w = 0; w < W; ++w) v[k] = max(v[k], red[w * K + k]);
  }
}
// whether all groups that share this warp or CTA say yes (groups of a warp or more: uniform already)
template <int N>
__device__ __forceinline__ bool grp_all(bool yes) {
  if constexpr (Grp<N>::T < 32) return __all_sync(0xffffffffu, yes);
  else return yes;
}

// a shared cell of 8 bytes holds a double or a split fixed-point value
using cell = long long;
__device__ __forceinline__ fx c_fx(cell c) { return {(int)(c >> 32), (int)c}; }
__device__ __forceinline__ cell c_of(fx x) { return ((long long)x.hi << 32) | (unsigned)x.lo; }
template <int LH>
__device__ __forceinline__ cell c_split(long long X) { return c_of(fx_split<LH>(X)); }
__device__ __forceinline__ double c_d(cell c) { return __longlong_as_double(c); }
__device__ __forceinline__ cell c_of(double d) { return __double_as_longlong(d); }

// operators in shared memory: fixed point and, for the FP64 twins, double
template <int N>
struct XOps {
  cell B[N * N], Bt[N * N], Dn[N * N], lift[2][N], end[2][N];
  double dB[N * N], dBt[N * N], dDh[N * N], de[2][N], deh[2][N];
};
template <int N>
__device__ __forceinline__ void load_xops(const Ops* __restrict__ o, XOps<N>& s) {
  auto pack = [](int2 v) { return c_of(fx{v.x, v.y}); };
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) {
    s.B[i] = pack(o->xB[i]);
    s.Bt[i] = pack(o->xBt[i]);
    s.Dn[i] = pack(o->xDn[i]);
    s.dB[i] = o->B[i];
    s.dBt[i] = o->Bt[i];
    s.dDh[i] = o->Dh[i];
  }
  for (int i = threadIdx.x; i < 2 * N; i += blockDim.x) {
    const int side = i / N, k = i % N;
    s.lift[side][k] = pack(o->xlift[side][k]);
    s.end[side][k] = pack(o->xend[side][k]);
    s.de[side][k] = side ? o->eR[k] : o->eL[k];
    s.deh[side][k] = o->eh[side][k];
  }
  __syncthreads();
}

// volume points behind face point f of face phi: base + k * stride
template <int N>
__device__ __forceinline__ void face_line(int phi, int f, int& base, int& st) {
  const int is = f % N, it = f / N, axis = phi >> 1;
  base = axis == 0 ? N * f : axis == 1 ? is + N * N * it : f;
  st = axis == 0 ? 1 : axis == 1 ? N : N * N;
}

// one pass of C fields along direction DIR at point g: out = A in (T: A^T in), data split at 30 bits
template <int N, int DIR, bool TR, bool FX, int C>
__device__ __forceinline__ void pass_b(const XOps<N>& so, const cell* in, cell* out, int g) {
  constexpr int NP = N * N * N, ST = DIR == 0 ? 1 : DIR == 1 ? N : N * N;
  const int i = (g / ST) % N, base = g - i * ST;
  if constexpr (FX) {
    fx a[N];
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] = c_fx(TR ? so.Bt[k * N + i] : so.B[i * N + k]);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      fxacc s = fx_zero<30>();
#pragma unroll
      for (int k = 0; k < N; ++k) fx_mac(s, a[k], c_fx(in[c * NP + base + k * ST]));
      out[c * NP + g] = c_split<30>(fx_sum<30>(s));
    }
  } else {
    for (int c = 0; c < C; ++c) {
      double s = 0.0;
      for (int k = 0; k < N; ++k) s = fma(TR ? so.dBt[k * N + i] : so.dB[i * N + k], c_d(in[c * NP + base + k * ST]), s);
      out[c * NP + g] = c_of(s);
    }
  }
}

// --------------------------------------------------------------------------------------------
// nodal values -> Gauss values and face traces
// --------------------------------------------------------------------------------------------
template <int N, bool FX>
__device__ __forceinline__ void interp_body(const XOps<N>& so, const double (&x)[5], const int (&ex)[5], cell* b0,
                                            cell* b1, int g, bool act, bool live, int row, double* __restrict__ ug,
                                            double* __restrict__ uf) {
  constexpr int NP = Grp<N>::NP, NF = Grp<N>::NF, T = Grp<N>::T;
  if (act)
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if constexpr (FX) b0[c * NP + g] = c_split<30>(fx_from<59>(x[c], ex[c]));
      else b0[c * NP + g] = c_of(x[c]);
    }
  grp_sync<N>();
  if (act) pass_b<N, 0, false, FX, 5>(so, b0, b1, g);
  grp_sync<N>();
  if (act) pass_b<N, 1, false, FX, 5>(so, b1, b0, g);
  grp_sync<N>();
  if (act) pass_b<N, 2, false, FX, 5>(so, b0, b1, g);
  grp_sync<N>();
  if (!live) return;
  if (act)
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const cell v = b1[c * NP + g];
      if constexpr (FX) {
        ug[c * NP + g] = fx_to_double(fx_join<30>(c_fx(v)), ex[c] - 1081);
      } else {
        ug[c * NP + g] = c_d(v);
      }
    }
  for (int idx = g; idx < 6 * NF; idx += T) {
    const int phi = idx / NF, f = idx % NF;
    int base, st;
    face_line<N>(phi, f, base, st);
    double out[5];
    if constexpr (FX) {
      fxacc s[5] = {fx_zero<30>(), fx_zero<30>(), fx_zero<30>(), fx_zero<30>(), fx_zero<30>()};
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const fx ev = c_fx(so.end[phi & 1][k]);
#pragma unroll
        for (int c = 0; c < 5; ++c) fx_mac(s[c], ev, c_fx(b1[c * NP + base + k * st]));
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) out[c] = fx_to_double(fx_sum<30>(s[c]), ex[c] - 1081);
    } else {
      for (int c = 0; c < 5; ++c) {
        out[c] = 0.0;
        for (int k = 0; k < N; ++k) out[c] = fma(so.de[phi & 1][k], c_d(b1[c * NP + base + k * st]), out[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) uf[(phi * row + c) * NF + f] = out[c];
  }
}
template <int N>
__device__ __noinline__ void interp_slow(const XOps<N>& so, const double (&x)[5], const int (&ex)[5], cell* b0, cell* b1,
                                         int g, bool act, bool live, int row, double* ug, double* uf) {
  interp_body<N, false>(so, x, ex, b0, b1, g, act, live, row, ug, uf);
}

// GRAD = false: plane blockIdx.y, u -> value plane, v -> tangent plane of ug, uf (grid.y = 1: u alone).
// GRAD = true: a nodal gradient u [E][3][5][NP], direction blockIdx.y, to ug [E][3][5][NP], uf [E][6][15][NF].
template <int N, bool GRAD>
__global__ void __launch_bounds__(128) k_interp64(const double* __restrict__ u, const double* __restrict__ v,
                                                  long long E, const Ops* __restrict__ ops, double* __restrict__ ug,
                                                  double* __restrict__ uf) {
  constexpr int NP = Grp<N>::NP, NF = Grp<N>::NF, T = Grp<N>::T;
  constexpr int ROW = GRAD ? 15 : 5;         // variables of an element's record
  __shared__ XOps<N> so;
  __shared__ int red[5 * 4];
  extern __shared__ __align__(16) cell cells[];
  load_xops<N>(ops, so);
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  cell* b0 = cells + grp * 10 * NP;
  const long long e = (long long)blockIdx.x * (blockDim.x / T) + grp;
  const bool live = e < E, act = g < NP;
  const int c0 = GRAD ? 5 * blockIdx.y : 0;
  const double* in = (!GRAD && blockIdx.y ? v : u) + (e * ROW + c0) * NP;
  double x[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  int ex[5];
  if (live && act)
#pragma unroll
    for (int c = 0; c < 5; ++c) x[c] = in[c * NP + g];
#pragma unroll
  for (int c = 0; c < 5; ++c) ex[c] = fx_mag(x[c]);
  grp_max<N, 5>(ex, red);
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    ok = ok && fx_ok(ex[c]);
    ex[c] = fx_exp(ex[c]);
  }
  const long long pl = !GRAD && blockIdx.y ? E : 0;
  double* go = ug + ((pl + e) * ROW + c0) * NP;
  double* fo = uf + ((pl + e) * 6 * ROW + c0) * NF;
  if (!grp_all<N>(ok)) {
    interp_slow<N>(so, x, ex, b0, b0 + 5 * NP, g, act, live && !ok, ROW, go, fo);
    if constexpr (T >= 32) return;
    grp_sync<N>();                           // groups of this warp that passed take the fixed-point path
  }
  interp_body<N, true>(so, x, ex, b0, b0 + 5 * NP, g, act, live && ok, ROW, go, fo);
}

// --------------------------------------------------------------------------------------------
// products with the element mass matrix M = B^T W B and its inverse, and Gauss values -> nodal values
// --------------------------------------------------------------------------------------------
// Each is two or one sum-factorised transforms of the five variables (MODE 2: of one direction of the
// gradient), bound by shared-memory loads and the integer pipe instead of the FP64 pipe (12,288 elements,
// p = 2: mass 73 us, inverse 60 us with FP64 passes).
enum { NODAL_MASS = 0, NODAL_MASS_INV = 1, NODAL_FROM_GAUSS = 2 };

// one pass with an operator given by its fixed-point (cx) and FP64 (cd) coefficients
template <int N, int DIR, bool TR, bool FX>
__device__ __forceinline__ void pass_c(const cell* cx, const double* cd, const cell* in, cell* out, int g) {
  constexpr int NP = N * N * N, ST = DIR == 0 ? 1 : DIR == 1 ? N : N * N;
  const int i = (g / ST) % N, base = g - i * ST;
  if constexpr (FX) {
    fx a[N];
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] = c_fx(cx[TR ? k * N + i : i * N + k]);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      fxacc s = fx_zero<30>();
#pragma unroll
      for (int k = 0; k < N; ++k) fx_mac(s, a[k], c_fx(in[c * NP + base + k * ST]));
      out[c * NP + g] = c_split<30>(fx_sum<30>(s));
    }
  } else {
    for (int c = 0; c < 5; ++c) {
      double s = 0.0;
      for (int k = 0; k < N; ++k) s = fma(cd[TR ? k * N + i : i * N + k], c_d(in[c * NP + base + k * ST]), s);
      out[c * NP + g] = c_of(s);
    }
  }
}
// three passes, from b0 into b1
template <int N, bool TR, bool FX>
__device__ __forceinline__ void transform(const cell* cx, const double* cd, cell* b0, cell* b1, int g, bool act) {
  grp_sync<N>();
  if (act) pass_c<N, 0, TR, FX>(cx, cd, b0, b1, g);
  grp_sync<N>();
  if (act) pass_c<N, 1, TR, FX>(cx, cd, b1, b0, g);
  grp_sync<N>();
  if (act) pass_c<N, 2, TR, FX>(cx, cd, b0, b1, g);
  grp_sync<N>();
}

template <int N>
struct NodalOps {
  cell B[N * N], Bt[N * N], Binv[N * N];
  double dB[N * N], dBt[N * N], dBinv[N * N], iw[N];
};

template <int N, int MODE>
__device__ __noinline__ void nodal_slow(const NodalOps<N>& so, double (&x)[5], double factor, cell* b0, cell* b1, int g,
                                        bool act) {
  constexpr int NP = N * N * N;
  auto put = [&](double f) {
    if (act)
      for (int c = 0; c < 5; ++c) b0[c * NP + g] = c_of(x[c] * f);
  };
  auto get = [&]() {
    if (act)
      for (int c = 0; c < 5; ++c) x[c] = c_d(b1[c * NP + g]);
  };
  put(1.0);
  if constexpr (MODE == NODAL_MASS) transform<N, false, false>(nullptr, so.dB, b0, b1, g, act);
  if constexpr (MODE == NODAL_MASS_INV) transform<N, true, false>(nullptr, so.dBinv, b0, b1, g, act);
  if constexpr (MODE != NODAL_FROM_GAUSS) {
    get();
    put(factor);
  }
  if constexpr (MODE == NODAL_MASS) transform<N, true, false>(nullptr, so.dBt, b0, b1, g, act);
  else transform<N, false, false>(nullptr, so.dBinv, b0, b1, g, act);
  get();
}

// in and out [E][ROW][NP] (they may be the same array); NODAL_FROM_GAUSS: direction blockIdx.y of [E][3][5][NP]
template <int N, int MODE>
__global__ void __launch_bounds__(128) k_nodal64(long long E, const Ops* __restrict__ ops, const double* in_g,
                                                 double* out_g, const double* __restrict__ gu) {
  constexpr int NP = Grp<N>::NP, T = Grp<N>::T;
  constexpr int ROW = MODE == NODAL_FROM_GAUSS ? 15 : 5;
  __shared__ NodalOps<N> so;
  __shared__ int red[6 * 4];
  extern __shared__ __align__(16) cell cells[];
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) {
    so.B[i] = c_of(fx{ops->xB[i].x, ops->xB[i].y});
    so.Bt[i] = c_of(fx{ops->xBt[i].x, ops->xBt[i].y});
    so.Binv[i] = c_of(fx{ops->xBinv[i].x, ops->xBinv[i].y});
    so.dB[i] = ops->B[i];
    so.dBt[i] = ops->Bt[i];
    so.dBinv[i] = ops->Binv[i];
  }
  for (int i = threadIdx.x; i < N; i += blockDim.x) so.iw[i] = ops->iw[i];
  __syncthreads();
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  cell *b0 = cells + grp * 10 * NP, *b1 = b0 + 5 * NP;
  const long long e = (long long)blockIdx.x * (blockDim.x / T) + grp;
  const bool live = e < E, act = g < NP;
  const long long at = (e * ROW + (MODE == NODAL_FROM_GAUSS ? 5 * blockIdx.y : 0)) * NP + g;
  double x[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, factor = 1.0;
  int mx[6] = {0, 0, 0, 0, 0, 0};
  if (live && act) {
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      x[c] = in_g[at + c * NP];
      mx[c] = fx_mag(x[c]);
    }
    if constexpr (MODE == NODAL_MASS) factor = gu[e * 11 * NP + 9 * NP + g];
    if constexpr (MODE == NODAL_MASS_INV)
      factor = gu[e * 11 * NP + 10 * NP + g] * (so.iw[g % N] * so.iw[(g / N) % N] * so.iw[g / (N * N)]);
    mx[5] = fx_mag(factor);
  }
  grp_max<N, 6>(mx, red);
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    ok = ok && fx_ok(mx[c]);
    mx[c] = fx_exp(mx[c]);
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) ok = ok && mx[c] + mx[5] >= 1300 && mx[c] + mx[5] <= 2900;
  const bool slow = live && !ok;
  if (!grp_all<N>(ok)) {
    nodal_slow<N, MODE>(so, x, factor, b0, b1, g, act && slow);
    if (act && slow)
#pragma unroll
      for (int c = 0; c < 5; ++c) out_g[at + c * NP] = x[c];
    if constexpr (T >= 32) return;
    grp_sync<N>();
  }
  // data bits: the passes grow values by the operators' sums (B 2.7, Bt 2.4, Binv^T 16.1, Binv 36.7 for
  // three passes), and the splits hold 61 bits
  constexpr int BITS = MODE == NODAL_MASS ? 57 : MODE == NODAL_MASS_INV ? 56 : 55;
  int sh[5];                                 // exponent of a unit
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    sh[c] = mx[c] - BITS - 1022;
    if (act) b0[c * NP + g] = c_split<30>(fx_from<BITS>(x[c], mx[c]));
  }
  if constexpr (MODE == NODAL_MASS) transform<N, false, true>(so.B, nullptr, b0, b1, g, act);
  if constexpr (MODE == NODAL_MASS_INV) transform<N, true, true>(so.Binv, nullptr, b0, b1, g, act);
  if constexpr (MODE != NODAL_FROM_GAUSS) {
    const fx f = fx_split<27>(fx_from<57>(factor, mx[5]));
    long long y[5] = {0, 0, 0, 0, 0};
    int up[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      if (act) y[c] = fx_mul<30>(f, c_fx(b1[c * NP + g]));
      sh[c] += mx[5] - 1022;
      if constexpr (MODE == NODAL_MASS_INV) up[c] = 64 - __clzll(y[c] < 0 ? -y[c] : y[c]);
    }
    if constexpr (MODE == NODAL_MASS_INV) {
      grp_max<N, 5>(up, red);
#pragma unroll
      for (int c = 0; c < 5; ++c) {          // to 55 bits
        const int d = up[c] ? up[c] - 55 : 0;
        sh[c] += d;
        y[c] = d >= 0 ? (y[c] + (d ? 1LL << (d - 1) : 0LL)) >> d : y[c] << -d;
      }
    }
    if (act)
#pragma unroll
      for (int c = 0; c < 5; ++c) b0[c * NP + g] = c_split<30>(y[c]);
  }
  if constexpr (MODE == NODAL_MASS) transform<N, true, true>(so.Bt, nullptr, b0, b1, g, act);
  else transform<N, false, true>(so.Binv, nullptr, b0, b1, g, act);
  if (act && live && ok)
#pragma unroll
    for (int c = 0; c < 5; ++c) out_g[at + c * NP] = fx_to_double(fx_join<30>(c_fx(b1[c * NP + g])), sh[c]);
}

// --------------------------------------------------------------------------------------------
// LDG gradient (Eq. DGformulation a) in Gauss space and its face traces
// --------------------------------------------------------------------------------------------
// Shared cells of a group: sY [9][NP] G u of the current variable, sL [6][3][NF] n u_hat of the current
// variable, sN [3][6 NF] normals, sUh [5][6 NF] u_hat, sQ [3][NP] gradient of the current variable, sU [5][NP].
template <int N>
struct GradCells {
  static constexpr int NP = N * N * N, NF = N * N;
  static constexpr int Y = 0, L = Y + 9 * NP, Nn = L + 18 * NF, Uh = Nn + 18 * NF, Q = Uh + 30 * NF, U = Q + 3 * NP,
                       size = U + 5 * NP;
  // the sum of at most 2^57 times the operators' column sums, shifted to stay below 2^61
  static constexpr int SH = N == 2 ? 0 : N == 3 ? 1 : 2;
};

// the FP64 twin of k_grad64's loop (sN, sUh, sU hold doubles)
template <int N>
__device__ __noinline__ void grad_slow(const XOps<N>& so, const double* gu, cell* cells, int g, bool act, bool live,
                                       double* qg, double* qf) {
  using C = GradCells<N>;
  constexpr int NP = C::NP, NF = C::NF, T = Grp<N>::T;
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  for (int c = 0; c < 5; ++c) {
    if (act && live)
      for (int k = 0; k < 9; ++k) cells[C::Y + k * NP + g] = c_of(gu[k * NP + g] * c_d(cells[C::U + c * NP + g]));
    for (int idx = g; idx < 6 * NF; idx += T)
      for (int d = 0; d < 3; ++d)
        cells[C::L + (idx / NF * 3 + d) * NF + idx % NF] =
            c_of(c_d(cells[C::Nn + d * 6 * NF + idx]) * c_d(cells[C::Uh + c * 6 * NF + idx]));
    grp_sync<N>();
    if (act && live)
      for (int d = 0; d < 3; ++d) {
        double s = 0.0;
        for (int a = 0; a < 3; ++a) {
          const int st = a == 0 ? 1 : a == 1 ? N : N * N;
          const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
          for (int side = 0; side < 2; ++side)
            s = fma(so.deh[side][i], c_d(cells[C::L + ((2 * a + side) * 3 + d) * NF + fp]), s);
          for (int k = 0; k < N; ++k) s = fma(-so.dDh[k * N + i], c_d(cells[C::Y + (a * 3 + d) * NP + base + k * st]), s);
        }
        s *= gu[10 * NP + g];
        cells[C::Q + d * NP + g] = c_of(s);
        qg[(d * 5 + c) * NP + g] = s;
      }
    grp_sync<N>();
    if (live)
      for (int idx = g; idx < 6 * NF; idx += T) {
        const int phi = idx / NF, f = idx % NF;
        int base, st;
        face_line<N>(phi, f, base, st);
        for (int d = 0; d < 3; ++d) {
          double s = 0.0;
          for (int k = 0; k < N; ++k) s = fma(so.de[phi & 1][k], c_d(cells[C::Q + d * NP + base + k * st]), s);
          qf[(phi * 15 + d * 5 + c) * NF + f] = s;
        }
      }
    grp_sync<N>();
  }
}

// plane plane0 + blockIdx.y of qg, qf from the same plane of ug, uf (0: value, 1: tangent). The wall
// trace of the tangent reads the value plane's varrho trace.
template <int N>
__global__ void __launch_bounds__(128, 5) k_grad64(long long E, const Ops* __restrict__ ops, double t_wall, int plane0,
                                                const double* __restrict__ gu, const double* __restrict__ fgu,
                                                const int* __restrict__ nbr, const int* __restrict__ nbr_fo,
                                                const double* __restrict__ ug, const double* __restrict__ uf,
                                                double* __restrict__ qg, double* __restrict__ qf) {
  using C = GradCells<N>;
  constexpr int NP = Grp<N>::NP, NF = Grp<N>::NF, T = Grp<N>::T, NI = Grp<N>::NI, SH = C::SH;
  __shared__ XOps<N> so;
  __shared__ int red[9 * 4];
  extern __shared__ __align__(16) cell cells_all[];
  load_xops<N>(ops, so);
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  cell* cells = cells_all + (size_t)grp * C::size;
  cell *sY = cells + C::Y, *sL = cells + C::L, *sN = cells + C::Nn, *sUh = cells + C::Uh, *sQ = cells + C::Q,
       *sU = cells + C::U;
  const long long e = (long long)blockIdx.x * (blockDim.x / T) + grp;
  bool live = e < E;
  const bool act = g < NP;
  const int plane = plane0 + blockIdx.y;
  const double* ufp = uf + plane * E * 30 * NF;
  const double* gue = gu + e * 11 * NP;
  int mx[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};   // geometry per d, field per c, 1 / |J|
  if (live && act) {
    const double* ugp = ug + (plane * E + e) * 5 * NP;
#pragma unroll
    for (int k = 0; k < 9; ++k) mx[k % 3] = max(mx[k % 3], fx_mag(gue[k * NP + g]));
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const double u = ugp[c * NP + g];
      sU[c * NP + g] = c_of(u);
      mx[3 + c] = fx_mag(u);
    }
    mx[8] = fx_mag(gue[10 * NP + g]);
  }
  // traces u_hat (Eq. LDG2) and face geometry, as doubles until the exponents are known
#pragma unroll
  for (int it = 0; it < NI; ++it) {
    const int idx = g + it * T;
    if (!live || idx >= 6 * NF) continue;
    const int phi = idx / NF, f = idx % NF;
    const long long fbase = e * 30 * NF + phi * 5 * NF + f;
    const int nb = nbr[e * 6 + phi];
    double uh[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) uh[c] = ufp[fbase + c * NF];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const double n = fgu[((e * 6 + phi) * 4 + d) * NF + f];
      sN[d * 6 * NF + idx] = c_of(n);
      mx[d] = max(mx[d], fx_mag(n));
    }
    if (nb >= 0) {
      const int fo = nbr_fo[e * 6 + phi];
      const int f2 = orient_map(fo >> 3, f % N, f / N, N);
      const long long nbase = (long long)nb * 30 * NF + (fo & 7) * 5 * NF + f2;
      double oth[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) oth[c] = ufp[nbase + c * NF];
#pragma unroll
      for (int c = 0; c < 5; ++c) uh[c] = 0.5 * (uh[c] + oth[c]);
    } else if (nb == -DG_BC_WALL) {
      const double sr = exp_fast(0.5 * uf[fbase]);   // the value plane's varrho trace
      uh[1] = uh[2] = uh[3] = 0.0;
      uh[4] = plane == 0 ? sr * t_wall : 0.5 * sr * t_wall * uh[0];
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      sUh[c * 6 * NF + idx] = c_of(uh[c]);
      mx[3 + c] = max(mx[3 + c], fx_mag(uh[c]));
    }
  }
  grp_max<N, 9>(mx, red);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    ok = ok && fx_ok(mx[k]);
    mx[k] = fx_exp(mx[k]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const int s = mx[d] + mx[3 + c] + mx[8];
      ok = ok && s >= 2200 && s <= 3980;
    }
  double* qge = qg + (plane * E + e) * 15 * NP;
  double* qfe = qf + (plane * E + e) * 90 * NF;
  if (!grp_all<N>(ok)) {
    grad_slow<N>(so, gue, cells, g, act, live && !ok, qge, qfe);
    if constexpr (T >= 32) return;
  }
  live = live && ok;
  // fixed point: own entries, so no barrier is needed
  fx G[9], wx{0, 0};
  if (live && act) {
#pragma unroll
    for (int k = 0; k < 9; ++k) G[k] = fx_split<29>(fx_from<57>(gue[k * NP + g], mx[k % 3]));
    wx = fx_split<27>(fx_from<57>(gue[10 * NP + g], mx[8]));
#pragma unroll
    for (int c = 0; c < 5; ++c) sU[c * NP + g] = c_split<28>(fx_from<58>(c_d(sU[c * NP + g]), mx[3 + c]));
  }
  int lofs[NI], tb[NI], ts[NI], qo[NI];
#pragma unroll
  for (int it = 0; it < NI; ++it) {
    const int idx = g + it * T;
    const int phi = idx / NF, f = idx % NF;
    lofs[it] = live && idx < 6 * NF ? phi * 3 * NF + f : -1;
    qo[it] = phi * 15 * NF + f;
    face_line<N>(phi, f, tb[it], ts[it]);
    if (lofs[it] < 0) continue;
#pragma unroll
    for (int d = 0; d < 3; ++d) sN[d * 6 * NF + idx] = c_split<29>(fx_from<57>(c_d(sN[d * 6 * NF + idx]), mx[d]));
#pragma unroll
    for (int c = 0; c < 5; ++c) sUh[c * 6 * NF + idx] = c_split<28>(fx_from<58>(c_d(sUh[c * 6 * NF + idx]), mx[3 + c]));
  }
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  int ec = mx[3];
#pragma unroll 1
  for (int c = 0; c < 5; ++c) {
    // products: G u at the Gauss points, n u_hat at the face points
    if (live && act) {
      const fx ux = c_fx(sU[c * NP + g]);
#pragma unroll
      for (int k = 0; k < 9; ++k) sY[k * NP + g] = c_split<28>(fx_mul<28>(G[k], ux));
    }
#pragma unroll
    for (int it = 0; it < NI; ++it) {
      if (lofs[it] < 0) continue;
      const int idx = g + it * T;
      const fx uh = c_fx(sUh[c * 6 * NF + idx]);
#pragma unroll
      for (int d = 0; d < 3; ++d) sL[lofs[it] + d * NF] = c_split<28>(fx_mul<28>(c_fx(sN[d * 6 * NF + idx]), uh));
    }
    grp_sync<N>();
    const int sh = ec + mx[8] - 3123 + SH;
    if (act) {
      // q_d = (sum over the 6 faces of eh_face[i_axis] n_d u_hat_c - Dh^T (G u_c)) / |J|
      fxacc s[3] = {fx_zero<28>(), fx_zero<28>(), fx_zero<28>()};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int st = a == 0 ? 1 : a == 1 ? N : N * N;
        const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const fx ev = c_fx(so.lift[side][i]);
#pragma unroll
          for (int d = 0; d < 3; ++d) fx_mac(s[d], ev, c_fx(sL[((2 * a + side) * 3 + d) * NF + fp]));
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const fx D = c_fx(so.Dn[k * N + i]);
#pragma unroll
          for (int d = 0; d < 3; ++d) fx_mac(s[d], D, c_fx(sY[(a * 3 + d) * NP + base + k * st]));
        }
      }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const long long q = fx_mul<30>(wx, fx_split<30>(fx_sum<28>(s[d]) >> SH));
        sQ[d * NP + g] = c_split<30>(q);
        if (live) qge[(d * 5 + c) * NP + g] = fx_to_double(q, mx[d] + sh);
      }
    }
    grp_sync<N>();
#pragma unroll
    for (int it = 0; it < NI; ++it) {
      if (lofs[it] < 0) continue;
      const int side = ((g + it * T) / NF) & 1;
      fxacc s[3] = {fx_zero<30>(), fx_zero<30>(), fx_zero<30>()};
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const fx ev = c_fx(so.end[side][k]);
#pragma unroll
        for (int d = 0; d < 3; ++d) fx_mac(s[d], ev, c_fx(sQ[d * NP + tb[it] + k * ts[it]]));
      }
#pragma unroll
      for (int d = 0; d < 3; ++d)
        qfe[qo[it] + (d * 5 + c) * NF] = fx_to_double(fx_sum<30>(s[d]), mx[d] + sh);
    }
    ec = c == 0 ? mx[4] : c == 1 ? mx[5] : c == 2 ? mx[6] : mx[7];
  }
}

// The gradient trace that an element gets at a face from its neighbour's perturbation alone is
// kn(f) u_dot_nb(f): kn = kappa (w n dS) / 2 with kappa(f) = sum_k e_face[k]^2 / (w |J|)(g(f, k)).
template <int N>
__global__ void k_cross_kappa(long long E, const Ops* __restrict__ ops, const double* __restrict__ geo,
                              const double* __restrict__ fgeo, double* __restrict__ kn) {
  constexpr int NP = N * N * N, NF = N * N;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= E * 6 * NF) return;
  const long long e = i / (6 * NF);
  const int phi = (int)(i / NF % 6), f = (int)(i % NF);
  const double* ev = (phi & 1) ? ops->eR : ops->eL;
  double kappa = 0.0;
  for (int k = 0; k < N; ++k) kappa += ev[k] * ev[k] / geo[e * 10 * NP + 9 * NP + face_vol_point<N>(phi, f, k)];
  for (int d = 0; d < 3; ++d)
    kn[((e * 6 + phi) * 3 + d) * NF + f] = 0.5 * kappa * fgeo[((e * 6 + phi) * 4 + d) * NF + f];
}

// --------------------------------------------------------------------------------------------
// numerical flux of Eq. LDG2 on every face (without the face weights), written for both element faces
// --------------------------------------------------------------------------------------------
// F_hat . n = (F(u, q) + F(u2, q2)) . n / 2 + sigma(u_hat) (u - u_hat) |n| inside,
// F(u_b, q) . n + sigma(u_b) (u - u_b) |n| at a wall, F_inviscid(u) . n at an outflow face.
template <int N, int NC>
__global__ void __launch_bounds__(128, 3) k_faces64(long long E, long long F, PhysT<double> P,
                                                 const int* __restrict__ face_e, const int* __restrict__ face_f,
                                                 const int* __restrict__ nbr, const int* __restrict__ nbr_fo,
                                                 const double* __restrict__ fgu, const double* __restrict__ uf,
                                                 const double* __restrict__ qf, double* __restrict__ fh,
                                                 const double* __restrict__ mixf) {
  using S = typename std::conditional<NC == 2, D64, double>::type;
  constexpr int NF = N * N;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= F * NF) return;
  const long long fi = idx / NF;
  const int f = (int)(idx % NF);
  const long long e = face_e[fi];
  const int phi = face_f[fi];
  Mix<double> mx{P.cv, 1.0};
  if (P.comp) {   // mixture at this face point: [E][6][2][NF] = (c_v*, conductivity factor)
    mx.cv = mixf[((e * 6 + phi) * 2) * NF + f];
    mx.kfac = mixf[((e * 6 + phi) * 2 + 1) * NF + f];
  }
  const double pc = P.comp ? mx.cv * P.inv_gamma : P.p_coef;
  const long long plane_u = E * 30 * NF, plane_q = E * 90 * NF;
  const double* gp = fgu + ((e * 6 + phi) * 4) * NF + f;
  const double n[3] = {gp[0], gp[NF], gp[2 * NF]};
  const double area = gp[3 * NF];
  const long long ub = e * 30 * NF + phi * 5 * NF + f;
  const long long qb = e * 90 * NF + phi * 15 * NF + f;
  const int nb = nbr[e * 6 + phi];
  S u[5], out[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) u[c] = ld<S, NC, double>(uf + ub + c * NF, plane_u);
  auto grad_of = [&](long long base, S (&q)[3][5]) {
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int c = 0; c < 5; ++c) q[d][c] = ld<S, NC, double>(qf + base + (d * 5 + c) * NF, plane_q);
  };
  if (nb == -DG_BC_OUTFLOW) {
    const S s = s_isr(u[0]);
    flux_n64_inviscid(u, n, pc, s, out);
  } else {
    const bool wall = nb < 0;
    S ue[5];                                 // the state whose flux is taken: u, or the wall's
#pragma unroll
    for (int c = 0; c < 5; ++c) ue[c] = u[c];
    if (wall) {
      S s, sr;
      s_rho(u[0], s, sr);
      ue[1] = ue[2] = ue[3] = s_zero<S>();
      ue[4] = P.t_wall * sr;
    }
    {
      S q[3][5], s, K, K2;
      grad_of(qb, q);
      state64(P, ue, mx, s, K, K2);
      flux_n64(P, ue, q, n, pc, s, K, K2, out);
    }
    S ur[5];                                 // the jump's other state: the neighbour's, or the wall's
    S uh0 = ue[0], uh4 = ue[4];
    double weight = area;
    S f2v[5];
    long long ob2 = 0;
    if (!wall) {
      const int fo = nbr_fo[e * 6 + phi];
      const int phi2 = fo & 7;
      const int f2 = orient_map(fo >> 3, f % N, f / N, N);
      ob2 = (long long)nb * 30 * NF + phi2 * 5 * NF + f2;
      const long long qb2 = (long long)nb * 90 * NF + phi2 * 15 * NF + f2;
#pragma unroll
      for (int c = 0; c < 5; ++c) ur[c] = ld<S, NC, double>(uf + ob2 + c * NF, plane_u);
      S q[3][5], s, K, K2;
      grad_of(qb2, q);
      state64(P, ur, mx, s, K, K2);
      flux_n64(P, ur, q, n, pc, s, K, K2, f2v);
      uh0 = 0.5 * (u[0] + ur[0]);
      uh4 = 0.5 * (u[4] + ur[4]);
      weight = 0.5 * area;
    } else {
#pragma unroll
      for (int c = 0; c < 5; ++c) ur[c] = ue[c];
    }
    S sm, se;
    sigma64(P, uh0, uh4, mx, sm, se);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const S ju = weight * (u[c] - ur[c]);
      if (!wall) out[c] = 0.5 * (out[c] + f2v[c]);
      out[c] = c == 0 ? s_fma(P.lam, ju, out[c]) : s_fma(c == 4 ? se : sm, ju, out[c]);
      if (!wall) st(fh + ob2 + c * NF, plane_u, -out[c]);
    }
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) st(fh + ub + c * NF, plane_u, out[c]);
}

// --------------------------------------------------------------------------------------------
// pointwise flux and source, weak derivative, lifting of F_hat, B^T -> nodal r (and J v)
// --------------------------------------------------------------------------------------------
// the state at Gauss point g and its fluxes and sources (volume64), with the stage operator's mass term
template <int N, int NC, typename S>
__device__ __forceinline__ void volume_load(long long e, long long E, int g, const PhysT<double>& P, const Sun64& sun,
                                            const double* __restrict__ gu, const double* __restrict__ accg,
                                            const double* __restrict__ xg, const double* __restrict__ ug,
                                            const double* __restrict__ qg, const double* __restrict__ mixg,
                                            double inv_stage_c, S (&F)[12], S (&src)[5]) {
  constexpr int NP = N * N * N;
  const long long plane_g = E * 5 * NP, plane_q = E * 15 * NP;
  S u[5], q[3][5];
#pragma unroll
  for (int c = 0; c < 5; ++c) u[c] = ld<S, NC, double>(ug + e * 5 * NP + c * NP + g, plane_g);
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int c = 0; c < 5; ++c) q[d][c] = ld<S, NC, double>(qg + e * 15 * NP + (d * 5 + c) * NP + g, plane_q);
  const double det = gu[e * 11 * NP + 9 * NP + g];
  const double a3[3] = {accg[e * 3 * NP + g], accg[e * 3 * NP + NP + g], accg[e * 3 * NP + 2 * NP + g]};
  double x3[3] = {0.0, 0.0, 0.0};
  if (P.euv) {
    x3[0] = xg[e * 3 * NP + g];
    x3[1] = xg[e * 3 * NP + NP + g];
    x3[2] = xg[e * 3 * NP + 2 * NP + g];
  }
  double mg[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (P.comp) {
#pragma unroll
    for (int k = 0; k < 8; ++k) mg[k] = mixg[(e * 8 + k) * NP + g];
  }
  volume64<S>(P, u, q, det, a3, x3, sun, mg, F, src);
  if constexpr (NC == 2)
    if (inv_stage_c != 0.0) {
      const double w = -det * inv_stage_c;
#pragma unroll
      for (int c = 0; c < 5; ++c) src[c].d = fma(w, u[c].d, src[c].d);
    }
}
// component (c, d) of the fluxes in F
__device__ __forceinline__ constexpr int flux_index(int c, int d) {
  return c == 0 ? 6 + d : c == 4 ? 9 + d : c - 1 == d ? d : 2 + (c - 1) + d;
}
template <int NC, int PL, typename S>
__device__ __forceinline__ double plane_of(const S& x) {
  if constexpr (NC == 1) return x;
  else return PL == 0 ? x.v : x.d;
}

// Cells of a group: sF [NC][15][NP] (reference fluxes a * 5 + c), sS [NC][5][NP] (sources), sH [5][6 NF]
template <int N, int NC>
struct VolCells {
  static constexpr int NP = N * N * N, NF = N * N;
  static constexpr int S = NC * 15 * NP, H = S + NC * 5 * NP, size = H + 30 * NF;
};

// the FP64 twin of k_volume64 from the reference fluxes on: sF and sS hold doubles
template <int N, int NC>
__device__ __noinline__ void volume_slow(const XOps<N>& so, long long e, long long E, int g, bool act, bool own,
                                         const double* fh, double stage_c, int pl0, cell* cells, double* r, double* jv) {
  using C = VolCells<N, NC>;
  constexpr int NP = C::NP, NF = C::NF, T = Grp<N>::T;
  cell *sF = cells, *sS = cells + C::S, *sH = cells + C::H;
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  for (int pl = pl0; pl < NC; ++pl) {
    grp_sync<N>();
    if (own)
      for (int idx = g; idx < 6 * NF; idx += T)
        for (int c = 0; c < 5; ++c)
          sH[c * 6 * NF + idx] = c_of(fh[pl * E * 30 * NF + e * 30 * NF + (idx / NF * 5 + c) * NF + idx % NF]);
    grp_sync<N>();
    cell* F = sF + pl * 15 * NP;
    double R[5];
    if (act)
      for (int c = 0; c < 5; ++c) {
        double s = c_d(sS[(pl * 5 + c) * NP + g]);
        for (int a = 0; a < 3; ++a) {
          const int st = a == 0 ? 1 : a == 1 ? N : N * N;
          const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
          for (int k = 0; k < N; ++k) s = fma(so.dDh[k * N + i], c_d(F[(a * 5 + c) * NP + base + k * st]), s);
          for (int side = 0; side < 2; ++side) s = fma(-so.deh[side][i], c_d(sH[c * 6 * NF + (2 * a + side) * NF + fp]), s);
        }
        R[c] = s;
      }
    grp_sync<N>();
    if (act)
      for (int c = 0; c < 5; ++c) F[c * NP + g] = c_of(R[c]);
    grp_sync<N>();
    if (act) pass_b<N, 0, true, false, 5>(so, F, F + 5 * NP, g);
    grp_sync<N>();
    if (act) pass_b<N, 1, true, false, 5>(so, F + 5 * NP, F, g);
    grp_sync<N>();
    if (act) pass_b<N, 2, true, false, 5>(so, F, F + 5 * NP, g);
    if (act)
      for (int c = 0; c < 5; ++c) {
        const double x = c_d(F[(5 + c) * NP + g]);
        if (pl == 0 && r) r[(e * 5 + c) * NP + g] = x;
        if (pl == 1) jv[(e * 5 + c) * NP + g] = stage_c != 0.0 ? -stage_c * x : x;
      }
  }
}

// stage_c != 0 (NC = 2): the tangent output is the DIRK stage operator J_G v = M v - stage_c J_r v. It is
// formed as -stage_c (J_r v - M v / stage_c), with -|J| u_dot / stage_c added to the tangent's source.
// CTAs per SM: latency of the pointwise physics against spills (Jv of a 16x16x8 degree-4 shell: 3 CTAs 1144 us, 4
// 1078, 5 1150; r of a 21x21x9 degree-3 shell: 3 CTAs 736, 4 689, 5 657).
// The physics is evaluated once for the twin too: a point out of range forms its reference fluxes in FP64, the others
// convert their products when their element is refused (residual of 12,288 degree-2 elements with composition, every one
// refused: 1505 us, 2183 with a second evaluation; ordinary calls 0.4 to 2 % of this kernel for the branch).
template <int N, int NC>
__global__ void __launch_bounds__(128, NC == 2 ? 4 : 5)
    k_volume64(long long E, const Ops* __restrict__ ops, PhysT<double> P, Sun64 sun, const double* __restrict__ gu,
               const double* __restrict__ accg, const double* __restrict__ xg, const double* __restrict__ ug,
               const double* __restrict__ qg, const double* __restrict__ fh, double* __restrict__ r,
               double* __restrict__ jv, double stage_c, double inv_stage_c, const double* __restrict__ mixg) {
  using S = typename std::conditional<NC == 2, D64, double>::type;
  using C = VolCells<N, NC>;
  constexpr int NP = Grp<N>::NP, NF = Grp<N>::NF, T = Grp<N>::T;
  __shared__ XOps<N> so;
  __shared__ int red[NC * 5 * 4];
  extern __shared__ __align__(16) cell cells_all[];
  load_xops<N>(ops, so);
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  cell* cells = cells_all + (size_t)grp * C::size;
  cell *sF = cells, *sS = cells + C::S, *sH = cells + C::H;
  const long long e = (long long)blockIdx.x * (blockDim.x / T) + grp;
  bool live = e < E;
  const bool act = g < NP;
  // per plane and variable: exponent bound (|x| < 2^(m - 1022)) of the reference fluxes, sources and face
  // fluxes; BAD marks magnitudes for the FP64 twin
  constexpr int BAD = 1 << 20;
  int mx[NC * 5];
#pragma unroll
  for (int k = 0; k < NC * 5; ++k) mx[k] = 0;
  auto expo = [](int mag) { return mag == 0 ? 0 : fx_ok(mag) ? mag >> 20 : BAD; };
  const int pl0 = NC == 2 && !r ? 1 : 0;     // the tangent alone when r is not wanted
  int eG[3] = {0, 0, 0}, eF[NC][3] = {};          // this point's exponents: geometry rows, flux groups
  bool bad = false;                               // this point's reference fluxes are doubles
  if (live && act) {
    S F[12], src[5];
    volume_load<N, NC, S>(e, E, g, P, sun, gu, accg, xg, ug, qg, mixg, inv_stage_c, F, src);
    double Gd[9];
    const double* gp = gu + e * 11 * NP + g;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      Gd[k] = gp[k * NP];
      eG[k / 3] = max(eG[k / 3], fx_mag(Gd[k]));
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      bad = bad || !fx_ok(eG[a]);
      eG[a] = fx_exp(eG[a]);
    }
    auto flux_exps = [&](auto plc) {              // momentum, varrho, energy
      constexpr int PL = decltype(plc)::value;
      int m[3] = {0, 0, 0};
#pragma unroll
      for (int k = 0; k < 12; ++k) m[k < 6 ? 0 : k < 9 ? 1 : 2] = max(m[k < 6 ? 0 : k < 9 ? 1 : 2], fx_mag(plane_of<NC, PL>(F[k])));
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        bad = bad || !fx_ok(m[k]);
        eF[PL][k] = fx_exp(m[k]);
      }
    };
    if (NC == 1 || r) flux_exps(std::integral_constant<int, 0>{});
    if constexpr (NC == 2) flux_exps(std::integral_constant<int, 1>{});
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      sS[c * NP + g] = c_of(plane_of<NC, 0>(src[c]));
      if (NC == 2) sS[(5 + c) * NP + g] = c_of(plane_of<NC, NC - 1>(src[c]));
    }
    if (bad) {
      mx[0] = BAD;
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          S x = s_zero<S>();
#pragma unroll
          for (int d = 0; d < 3; ++d) x = s_fma(Gd[a * 3 + d], F[flux_index(c, d)], x);
          sF[(a * 5 + c) * NP + g] = c_of(plane_of<NC, 0>(x));
          if (NC == 2) sF[(15 + a * 5 + c) * NP + g] = c_of(plane_of<NC, NC - 1>(x));
        }
    } else {
      fx G[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) G[k] = fx_split<29>(fx_from<58>(Gd[k], eG[k / 3]));
      // Fref[a][c] = sum_d G[a][d] F[c][d], exact to 2^-58 of this point's largest term of the row and group
      auto contract = [&](auto plc) {
        constexpr int PL = decltype(plc)::value;
        fx X[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) X[k] = fx_split<28>(fx_from<58>(plane_of<NC, PL>(F[k]), eF[PL][k < 6 ? 0 : k < 9 ? 1 : 2]));
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const int grp_c = c == 0 ? 1 : c == 4 ? 2 : 0;
          int ec = expo(fx_mag(plane_of<NC, PL>(src[c])));
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            fxacc s = fx_zero<28>();
#pragma unroll
            for (int d = 0; d < 3; ++d) fx_mac(s, G[a * 3 + d], X[flux_index(c, d)]);
            const long long R = fx_sum<28>(s);  // scale 2^(2103 - eG - eF)
            sF[(PL * 15 + a * 5 + c) * NP + g] = R;
            const int bits = 64 - __clzll(R < 0 ? -R : R);
            if (bits > 0) ec = max(ec, bits + eG[a] + eF[PL][grp_c] - 1081);
          }
          mx[PL * 5 + c] = ec;
        }
      };
      if (NC == 1 || r) contract(std::integral_constant<int, 0>{});
      if constexpr (NC == 2) contract(std::integral_constant<int, 1>{});
    }
  }
  const double* fhe = fh + e * 30 * NF;
  if (live)
    for (int pl = pl0; pl < NC; ++pl)
      for (int idx = g; idx < 6 * NF; idx += T) {
        const int phi = idx / NF, f = idx % NF;
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          const double h = fhe[pl * E * 30 * NF + (phi * 5 + c) * NF + f];
          if (pl == 0) {
            sH[c * 6 * NF + idx] = c_of(h);
            mx[c] = max(mx[c], expo(fx_mag(h)));
          } else {
            mx[NC * 5 - 5 + c] = max(mx[NC * 5 - 5 + c], expo(fx_mag(h)));
          }
        }
      }
  grp_max<N, NC * 5>(mx, red);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < NC * 5; ++k) {
    ok = ok && (mx[k] == 0 || (mx[k] >= 150 && mx[k] <= 1900));
    if (mx[k] == 0) mx[k] = 1023;
  }
  if (!grp_all<N>(ok)) {
    // the reference fluxes of the points that passed leave the fixed point (own entries)
    if (act && live && !ok && !bad)
      for (int pl = pl0; pl < NC; ++pl)
        for (int a = 0; a < 3; ++a)
          for (int c = 0; c < 5; ++c) {
            cell& x = sF[(pl * 15 + a * 5 + c) * NP + g];
            const int eFc = NC == 2 && pl == 1 ? eF[NC - 1][c == 0 ? 1 : c == 4 ? 2 : 0] : eF[0][c == 0 ? 1 : c == 4 ? 2 : 0];
            x = c_of(ldexp((double)x, eG[a] + eFc - 2103));
          }
    volume_slow<N, NC>(so, e, E, g, act && live && !ok, live && !ok, fh, stage_c, pl0, cells, r, jv);
    if constexpr (T >= 32) return;
  }
  live = live && ok;
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
#pragma unroll 1
  for (int pl = pl0; pl < NC; ++pl) {
    int ef[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) ef[c] = pl == 0 ? mx[c] : mx[NC * 5 - 5 + c];
    cell* Fp = sF + pl * 15 * NP;
    if (pl == 1 && live)                     // (the end of the value plane's pass left the sH reads behind)
      for (int idx = g; idx < 6 * NF; idx += T) {
        const int phi = idx / NF, f = idx % NF;
#pragma unroll
        for (int c = 0; c < 5; ++c)
          sH[c * 6 * NF + idx] = c_split<28>(fx_from<58>(fhe[E * 30 * NF + (phi * 5 + c) * NF + f], ef[c]));
      }
    if (pl == 0)
      for (int idx = g; idx < 6 * NF; idx += T)
#pragma unroll
        for (int c = 0; c < 5; ++c) {
          cell& x = sH[c * 6 * NF + idx];
          x = c_split<28>(fx_from<58>(c_d(x), ef[c]));
        }
    long long R[5] = {0, 0, 0, 0, 0};
    if (act) {
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        R[c] = (fx_from<58>(c_d(sS[(pl * 5 + c) * NP + g]), ef[c]) + 1) >> 1;
        const int grp_c = c == 0 ? 1 : c == 4 ? 2 : 0;
        const int eFc = (NC == 2 && pl == 1) ? eF[NC - 1][grp_c] : eF[0][grp_c];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          cell& x = Fp[(a * 5 + c) * NP + g];
          const int sh = ef[c] + 1023 - eG[a] - eFc;   // to |x| <= 2^58
          const long long y = sh < 0 ? x << min(-sh, 63) : x;
          const int rt = min(max(sh, 0), 63);
          x = c_split<28>((y >> rt) + ((rt ? y >> (rt - 1) : 0LL) & 1));
        }
      }
    }
    grp_sync<N>();
    if (act) {
      // minus the divergence part: -Dh^T F + eh F_hat, which the source subtracts
      fxacc s[5] = {fx_zero<28>(), fx_zero<28>(), fx_zero<28>(), fx_zero<28>(), fx_zero<28>()};
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int st = a == 0 ? 1 : a == 1 ? N : N * N;
        const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          const fx ev = c_fx(so.lift[side][i]);
#pragma unroll
          for (int c = 0; c < 5; ++c) fx_mac(s[c], ev, c_fx(sH[c * 6 * NF + (2 * a + side) * NF + fp]));
        }
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const fx D = c_fx(so.Dn[k * N + i]);
#pragma unroll
          for (int c = 0; c < 5; ++c) fx_mac(s[c], D, c_fx(Fp[(a * 5 + c) * NP + base + k * st]));
        }
      }
#pragma unroll
      for (int c = 0; c < 5; ++c) R[c] -= fx_sum<28>(s[c]);
    }
    // the sums nearly cancel (hydrostatic balance), so they keep three more bits than the bound on F
    // allows the passes of B^T, unless the largest of them needs those
    int up[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) up[c] = (int)((R[c] < 0 ? -R[c] : R[c]) >> 32);
    grp_max<N, 5>(up, red);
    grp_sync<N>();
    cell *b0 = Fp, *b1 = Fp + 5 * NP;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      up[c] = up[c] < (1 << 26) ? 0 : 6 - __clz(up[c]);
      if (act) b0[c * NP + g] = c_split<30>(R[c] >> up[c]);
    }
    grp_sync<N>();
    if (act) pass_b<N, 0, true, true, 5>(so, b0, b1, g);
    grp_sync<N>();
    if (act) pass_b<N, 1, true, true, 5>(so, b1, b0, g);
    grp_sync<N>();
    if (act) {
      pass_b<N, 2, true, true, 5>(so, b0, b1, g);
      if (live && (pl == 1 || r)) {
        double* out = (pl == 0 ? r : jv) + e * 5 * NP;
#pragma unroll
        for (int c = 0; c < 5; ++c) {        // own entries
          const double x = fx_to_double(fx_join<30>(c_fx(b1[c * NP + g])), ef[c] - 1079 + up[c]);
          out[c * NP + g] = (pl == 1 && stage_c != 0.0) ? -stage_c * x : x;
        }
      }
    }
  }
}

// --------------------------------------------------------------------------------------------
// launches
// --------------------------------------------------------------------------------------------
// threads per CTA: groups of a warp or less share a CTA of four warps once that still gives every SM
// several CTAs; with fewer elements one warp per CTA spreads them over all SMs (Jv, one warp against four per CTA:
// 3,072 degree-1 elements 113 against 122 us, 6,912 219 and 218, 98,304 2409 and 2279; degree 2, 1,536 elements 162.6
// and 163.3, 6,912 556 and 551, 98,304 6742 and 6616)
template <int N>
constexpr int groups64_max() { return Grp<N>::T > 32 ? 1 : 128 / Grp<N>::T; }   // groups of the largest CTA
template <int N>
inline int threads64(long long groups) {
  if constexpr (Grp<N>::T > 32) return Grp<N>::T;
  const long long warps = (groups * Grp<N>::T + 31) / 32;
  return warps <= NUM_SMS * 16 ? 32 : 128;
}

}  // namespace dg
