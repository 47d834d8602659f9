// Exact element diagonal blocks of the stage operator J_G = M - c J_r (FP64 arithmetic, FP32 storage).
//
// A column of an element's block is the response of its own residual to one of its own unit nodal values,
// including the path through its neighbours' LDG gradients. At a fixed state every step of that response is
// linear: interpolation of the unit value, the element's own gradient, a 20 x 20 Jacobian of the pointwise
// flux and source per Gauss point, a 5 x 20 Jacobian of the numerical flux per face point, weak derivative,
// lifting and projection. The neighbour answers through its gradient alone, whose trace at the shared face
// is kn(f) times the element's own trace (k_cross_kappa), so its part is folded into the face Jacobian's
// column. Evaluating the whole tangent of the residual for every one of the 5 (p+1)^3 unit values instead
// spent 99 % of its FP64 instructions on the same state (3,072 blocks of 135^2: 45.8 ms, of which faces and
// volume 35.7; now 8.7).
//   k_jac_volume  the volume Jacobians, twenty dual evaluations per point (1.4 ms)
//   k_jac_faces   the face Jacobians (0.7 ms)
//   k_blocks      all columns of one element per CTA: a unit value of variable c makes one variable's gradient
//                 (fixed point), 4 of the 20 Jacobian columns (80 + 20 FP64 FMAs per point and face point,
//                 the columns of variable c in shared memory) and the fixed-point contraction of k_volume64
//                 (6.5 ms, of which the Jacobian FMAs take 3.0 at the FP64 pipe's 2 per cycle and SM)
// Elements are processed in batches that bound the Jacobians' storage.
#pragma once

namespace dg {

template <int N>
struct Blk {
  static constexpr int NP = N * N * N, NF = N * N;
  // threads per column, columns in flight. k_blocks with half as many, these, twice as many: degree 1 (27,648 elements)
  // 6.15, 6.13, 10.4 ms; degree 2 (6,912) 20.8, 14.5, 15.1; degree 3 (1,296) 12.8, 12.6, 12.3; degree 4 (384) 26.4,
  // 19.3, 16.3. Two CTAs per SM fit at degree 2 (74 KB each), one at 3 and 4
  static constexpr int T = Grp<N>::T, GP = N <= 3 ? 8 : N == 4 ? 4 : 2;
  static constexpr long long JV = 400LL * NP, JF = 600LL * NF;               // doubles per element
  // cells of a column: gradient [9 + 3][NP] + [18][NF], then the reference fluxes [15][NP]; face fluxes [30][NF]
  static constexpr int W = 12 * NP + 18 * NF > 15 * NP ? 12 * NP + 18 * NF : 15 * NP;
  static constexpr int cells = 80 * NP + 20 * 6 * NF + 18 * NF + GP * (W + 30 * NF);
};

// direction dir of the 20: u_c (dir = c) or q_dc (dir = 5 + 5 d + c); rows: reference flux a * 5 + c, source 15 + c
template <int N>
__global__ void __launch_bounds__(128, 4) k_jac_volume(long long e0, long long nE, long long E, PhysT<double> P, Sun64 sun,
                                                    const double* __restrict__ gu, const double* __restrict__ accg,
                                                    const double* __restrict__ xg, const double* __restrict__ ug,
                                                    const double* __restrict__ qg, const double* __restrict__ mixg,
                                                    double* __restrict__ JV) {
  constexpr int NP = Blk<N>::NP;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nE * NP) return;
  const long long eb = i / NP, e = e0 + eb;
  const int g = (int)(i % NP);
  double x3[3] = {0.0, 0.0, 0.0}, mg[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  const double a3[3] = {accg[e * 3 * NP + g], accg[e * 3 * NP + NP + g], accg[e * 3 * NP + 2 * NP + g]};
  if (P.euv)
    for (int d = 0; d < 3; ++d) x3[d] = xg[e * 3 * NP + d * NP + g];
  if (P.comp)
    for (int k = 0; k < 8; ++k) mg[k] = mixg[(e * 8 + k) * NP + g];
  const double* gp = gu + e * 11 * NP + g;
  const double det = gp[9 * NP];
#pragma unroll 1
  for (int dir = 0; dir < 20; ++dir) {
    D64 u[5], q[3][5], F[12], src[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) u[c] = D64{ug[(e * 5 + c) * NP + g], dir == c ? 1.0 : 0.0};
#pragma unroll
    for (int k = 0; k < 15; ++k) q[k / 5][k % 5] = D64{qg[(e * 15 + k) * NP + g], dir == 5 + k ? 1.0 : 0.0};
    volume64<D64>(P, u, q, det, a3, x3, sun, mg, F, src);
    double* out = JV + (eb * 20 + dir) * 20 * NP + g;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double g0 = gp[(a * 3) * NP], g1 = gp[(a * 3 + 1) * NP], g2 = gp[(a * 3 + 2) * NP];
#pragma unroll
      for (int c = 0; c < 5; ++c)
        out[(a * 5 + c) * NP] = fma(g0, F[flux_index(c, 0)].d, fma(g1, F[flux_index(c, 1)].d, g2 * F[flux_index(c, 2)].d));
    }
#pragma unroll
    for (int c = 0; c < 5; ++c) out[(15 + c) * NP] = src[c].d;
  }
}

// Jacobian of an element's outward numerical flux (without face weights) at its face points with respect
// to its own traces: JF [eb][20 dir][5][6 NF]
template <int N>
__global__ void __launch_bounds__(128, 4) k_jac_faces(long long e0, long long nE, PhysT<double> P,
                                                   const int* __restrict__ nbr, const int* __restrict__ nbr_fo,
                                                   const double* __restrict__ fgu, const double* __restrict__ kn,
                                                   const double* __restrict__ uf, const double* __restrict__ qf,
                                                   const double* __restrict__ mixf, double* __restrict__ JF) {
  constexpr int NF = Blk<N>::NF;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nE * 6 * NF) return;
  const long long eb = i / (6 * NF), e = e0 + eb;
  const int phi = (int)(i / NF % 6), f = (int)(i % NF);
  const long long face = e * 6 + phi;
  const int nb = nbr[face];
  Mix<double> mx{P.cv, 1.0};
  if (P.comp) {
    mx.cv = mixf[(face * 2) * NF + f];
    mx.kfac = mixf[(face * 2 + 1) * NF + f];
  }
  const double pc = P.comp ? mx.cv * P.inv_gamma : P.p_coef;
  const double* gp = fgu + face * 4 * NF + f;
  const double n[3] = {gp[0], gp[NF], gp[2 * NF]};
  double* out = JF + eb * 600 * NF + phi * NF + f;
  double u[5], q[3][5];
#pragma unroll
  for (int c = 0; c < 5; ++c) u[c] = uf[(face * 5 + c) * NF + f];
#pragma unroll
  for (int k = 0; k < 15; ++k) q[k / 5][k % 5] = qf[(face * 15 + k) * NF + f];
  const bool wall = nb == -DG_BC_WALL, inner = nb >= 0;
  double u2[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, kn2[3] = {0.0, 0.0, 0.0}, Kb = 0.0, K2b = 0.0;
  if (inner) {
    const int fo = nbr_fo[face];
    const long long face2 = (long long)nb * 6 + (fo & 7);
    const int f2 = orient_map(fo >> 3, f % N, f / N, N);
#pragma unroll
    for (int c = 0; c < 5; ++c) u2[c] = uf[(face2 * 5 + c) * NF + f2];
#pragma unroll
    for (int d = 0; d < 3; ++d) kn2[d] = kn[(face2 * 3 + d) * NF + f2];
    double s2;
    state64(P, u2, mx, s2, Kb, K2b);
  }
  const double half = inner ? 0.5 : 1.0, weight = half * gp[3 * NF];
  double K = 0.0, K2 = 0.0;
  double ue[5];                              // the state whose flux is taken
#pragma unroll 1
  for (int c = 0; c < 5; ++c) {
    D64 ud[5], qd[3][5], F[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) ud[k] = D64{u[k], k == c ? 1.0 : 0.0};
#pragma unroll
    for (int k = 0; k < 15; ++k) qd[k / 5][k % 5] = D64{q[k / 5][k % 5], 0.0};
    double res[5];
    if (!inner && !wall) {
      flux_n64_inviscid(ud, n, pc, s_isr(ud[0]), F);
#pragma unroll
      for (int k = 0; k < 5; ++k) res[k] = F[k].d;
    } else {
      D64 ub[5], uh0, uh4, s, Kd, K2d, sm, se;
#pragma unroll
      for (int k = 0; k < 5; ++k) ub[k] = ud[k];
      if (wall) {
        D64 sw, sr;
        s_rho(ud[0], sw, sr);
        ub[1] = ub[2] = ub[3] = D64{0.0, 0.0};
        ub[4] = P.t_wall * sr;
        uh0 = ub[0];
        uh4 = ub[4];
      } else {
        uh0 = D64{0.5 * (u[0] + u2[0]), 0.5 * ud[0].d};
        uh4 = D64{0.5 * (u[4] + u2[4]), 0.5 * ud[4].d};
      }
      state64(P, ub, mx, s, Kd, K2d);
      flux_n64(P, ub, qd, n, pc, s, Kd, K2d, F);
      sigma64(P, uh0, uh4, mx, sm, se);
      K = Kd.v;
      K2 = K2d.v;
      double cross[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
      if (inner) {
        double dq[3][5];
#pragma unroll
        for (int k = 0; k < 15; ++k) dq[k / 5][k % 5] = k % 5 == c ? kn2[k / 5] : 0.0;
        flux_n64_dq(u2, dq, n, Kb, K2b, cross);
      }
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        ue[k] = ub[k].v;
        const double jump = u[k] - (wall ? ub[k].v : u2[k]);
        const double jd = ud[k].d - (wall ? ub[k].d : 0.0);
        const D64 sg = k == 0 ? D64{P.lam, 0.0} : k == 4 ? se : sm;
        res[k] = fma(half, F[k].d + cross[k], weight * fma(sg.d, jump, sg.v * jd));
      }
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) out[(c * 5 + k) * 6 * NF] = res[k];
  }
#pragma unroll 1
  for (int dc = 0; dc < 15; ++dc) {
    double dq[3][5], res[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 15; ++k) dq[k / 5][k % 5] = k == dc ? 1.0 : 0.0;
    if (inner || wall) flux_n64_dq(ue, dq, n, K, K2, res);
#pragma unroll
    for (int k = 0; k < 5; ++k) out[((5 + dc) * 5 + k) * 6 * NF] = half * res[k];
  }
}

// synchronisation of the T threads of column group grp inside a CTA that holds several
template <int N>
__device__ __forceinline__ void col_sync(int grp) {
  if constexpr (Grp<N>::T <= 32) __syncwarp();
  else asm volatile("bar.sync %0, %1;" ::"r"(grp + 1), "r"(Grp<N>::T) : "memory");
}
// grp_max for such a group; red: [W][K] of the group
template <int N, int K>
__device__ __forceinline__ void col_max(int (&v)[K], int* red, int grp) {
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
    const int warp = (threadIdx.x >> 5) % W;
    if ((threadIdx.x & 31) == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) red[warp * K + k] = v[k];
    col_sync<N>(grp);
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int w = 0; w < W; ++w) v[k] = max(v[k], red[w * K + k]);
  }
}

// One CTA per element, GP columns at a time. out [E][n][n] FP32, column-major blocks (n = 5 NP). jac false:
// the mass matrix alone (c = 0, given as stage_c = -1).
template <int N>
__global__ void __launch_bounds__(Blk<N>::GP * Blk<N>::T, N == 3 ? 2 : 1)
    k_blocks(long long e0, const Ops* __restrict__ ops, double t_wall, const double* __restrict__ gu,
             const double* __restrict__ fgu, const int* __restrict__ nbr, const double* __restrict__ uf,
             const double* __restrict__ JV, const double* __restrict__ JF, double stage_c, bool jac, float* __restrict__ out) {
  using B = Blk<N>;
  constexpr int NP = B::NP, NF = B::NF, T = B::T, GP = B::GP, NI = Grp<N>::NI, W = Grp<N>::W ? Grp<N>::W : 1;
  constexpr int SH = GradCells<N>::SH, n = 5 * NP;
  __shared__ XOps<N> so;
  __shared__ int red_all[GP][5 * W], bound[4];
  __shared__ double uw[6 * NF];              // d u_hat_4 / d varrho at wall face points, else 0
  extern __shared__ __align__(16) cell cells_all[];
  load_xops<N>(ops, so);
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  const bool act = g < NP;
  const long long eb = blockIdx.x, e = e0 + eb;
  double* VA = reinterpret_cast<double*>(cells_all);          // [4][20][NP] Jacobian columns u_c, q_0c, q_1c, q_2c
  double* FA = VA + 80 * NP;                                  // [4][5][6 NF]
  cell* sN = reinterpret_cast<cell*>(FA + 120 * NF);          // [3][6 NF] normals
  cell* work = sN + 18 * NF + (size_t)grp * (B::W + 30 * NF);
  cell *sY = work, *sL = sY + 9 * NP, *sQ = sL + 18 * NF;     // gradient of the column's variable
  cell* sF = work;                                            // [15][NP] reference fluxes, then the passes
  cell* sH = work + B::W;                                     // [5][6 NF]
  int* red = red_all[grp];
  const double* gue = gu + e * 11 * NP;
  // geometry exponents of the element (per direction d, and of 1 / |J|)
  if (threadIdx.x < 4) bound[threadIdx.x] = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < 9 * NP; i += blockDim.x) atomicMax(&bound[i / NP % 3], fx_mag(gue[i]));
  for (int i = threadIdx.x; i < NP; i += blockDim.x) atomicMax(&bound[3], fx_mag(gue[10 * NP + i]));
  for (int i = threadIdx.x; i < 18 * NF; i += blockDim.x) {
    const int d = i / (6 * NF), idx = i % (6 * NF);
    const double x = fgu[((e * 6 + idx / NF) * 4 + d) * NF + idx % NF];
    sN[i] = c_of(x);
    atomicMax(&bound[d], fx_mag(x));
  }
  bool has_wall = false;
  for (int phi = 0; phi < 6; ++phi) has_wall = has_wall || (jac && nbr[e * 6 + phi] == -DG_BC_WALL);
  for (int i = threadIdx.x; i < 6 * NF; i += blockDim.x)
    uw[i] = nbr[e * 6 + i / NF] == -DG_BC_WALL ? 0.5 * t_wall * exp_fast(0.5 * uf[(e * 6 + i / NF) * 5 * NF + i % NF]) : 0.0;
  __syncthreads();
  int eg[4];
  bool fx_geo = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    fx_geo = fx_geo && fx_ok(bound[k]);
    eg[k] = fx_exp(bound[k]);
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) fx_geo = fx_geo && eg[d] + eg[3] >= 1200 && eg[d] + eg[3] <= 2900;
  if (fx_geo)
    for (int i = threadIdx.x; i < 18 * NF; i += blockDim.x)
      sN[i] = c_split<29>(fx_from<57>(c_d(sN[i]), eg[i / (6 * NF)]));
  fx G[9], wx{0, 0};
  double det = 0.0;
  if (act) {
#pragma unroll
    for (int k = 0; k < 9; ++k) G[k] = fx_split<29>(fx_from<57>(gue[k * NP + g], eg[k % 3]));
    wx = fx_split<27>(fx_from<57>(gue[10 * NP + g], eg[3]));
    det = gue[9 * NP + g];
  }
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  const double inv_c = 1.0 / stage_c;
  int tb[NI], ts[NI];
#pragma unroll
  for (int it = 0; it < NI; ++it) {
    const int idx = g + it * T;
    face_line<N>(idx / NF, idx % NF, tb[it], ts[it]);
  }
#pragma unroll 1
  for (int c = 0; c < 5; ++c) {
    __syncthreads();
    for (int i = threadIdx.x; i < 80 * NP; i += blockDim.x) {
      const int k = i / (20 * NP);
      VA[i] = !jac ? 0.0 : JV[(eb * 20 + (k ? 5 * k + c : c)) * 20 * NP + i % (20 * NP)];
    }
    for (int i = threadIdx.x; i < 120 * NF; i += blockDim.x) {
      const int k = i / (30 * NF);
      FA[i] = !jac ? 0.0 : JF[(eb * 20 + (k ? 5 * k + c : c)) * 30 * NF + i % (30 * NF)];
    }
    __syncthreads();
    for (int b = grp; b < (NP + GP - 1) / GP * GP; b += GP) {
      // (every group runs the same number of columns; those beyond the last one write nothing)
      const bool live = b < NP;
      const int ib[3] = {b % N, (b / N) % N, b / (N * N) % N};
      // the unit value at the Gauss points, and its traces: l_b(-1), l_b(1) are 1 at the end nodes, else 0
      const double ud = act ? so.dB[ig[0] * N + ib[0]] * so.dB[ig[1] * N + ib[1]] * so.dB[ig[2] * N + ib[2]] : 0.0;
      double uft[NI], hat[NI];
#pragma unroll
      for (int it = 0; it < NI; ++it) {
        const int idx = g + it * T, phi = idx / NF, f = idx % NF, axis = phi >> 1;
        uft[it] = hat[it] = 0.0;
        if (idx >= 6 * NF) continue;
        const int is = f % N, itt = f / N;
        const int s_ax = axis == 0 ? 1 : 0, t_ax = axis == 2 ? 1 : 2;
        if (ib[axis] == ((phi & 1) ? N - 1 : 0)) uft[it] = so.dB[is * N + ib[s_ax]] * so.dB[itt * N + ib[t_ax]];
        const int nb = nbr[e * 6 + phi];
        hat[it] = nb >= 0 ? 0.5 * uft[it] : nb == -DG_BC_OUTFLOW ? uft[it] : c == 0 ? uft[it] : 0.0;
      }
      double qd[3] = {0.0, 0.0, 0.0}, qw[3] = {0.0, 0.0, 0.0};   // gradient of variable c; of 4 through the wall
      double qt[NI][3], qwt[NI][3];
      // gradient of `field` with traces `face` into q and its face traces
      auto gradient = [&](double field, const double (&face)[NI], double (&q)[3], double (&qtr)[NI][3]) {
        col_sync<N>(grp);
        if (fx_geo) {
          if (act) {
            const fx ux = fx_split<28>(fx_from<58>(field, 1023));     // both below 2
#pragma unroll
            for (int k = 0; k < 9; ++k) sY[k * NP + g] = c_split<28>(fx_mul<28>(G[k], ux));
          }
#pragma unroll
          for (int it = 0; it < NI; ++it) {
            const int idx = g + it * T;
            if (idx >= 6 * NF) continue;
            const fx uh = fx_split<28>(fx_from<58>(face[it], 1023));
#pragma unroll
            for (int d = 0; d < 3; ++d)
              sL[(idx / NF * 3 + d) * NF + idx % NF] = c_split<28>(fx_mul<28>(c_fx(sN[d * 6 * NF + idx]), uh));
          }
          col_sync<N>(grp);
          const int sh = 1023 + eg[3] - 3123 + SH;
          if (act) {
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
              const long long x = fx_mul<30>(wx, fx_split<30>(fx_sum<28>(s[d]) >> SH));
              sQ[d * NP + g] = c_split<30>(x);
              q[d] = fx_to_double(x, eg[d] + sh);
            }
          }
          col_sync<N>(grp);
#pragma unroll
          for (int it = 0; it < NI; ++it) {
            const int idx = g + it * T;
            if (idx >= 6 * NF) continue;
            const int side = (idx / NF) & 1;
            fxacc s[3] = {fx_zero<30>(), fx_zero<30>(), fx_zero<30>()};
#pragma unroll
            for (int k = 0; k < N; ++k) {
              const fx ev = c_fx(so.end[side][k]);
#pragma unroll
              for (int d = 0; d < 3; ++d) fx_mac(s[d], ev, c_fx(sQ[d * NP + tb[it] + k * ts[it]]));
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) qtr[it][d] = fx_to_double(fx_sum<30>(s[d]), eg[d] + sh);
          }
        } else {                             // FP64 twin
          if (act)
            for (int k = 0; k < 9; ++k) sY[k * NP + g] = c_of(gue[k * NP + g] * field);
#pragma unroll
          for (int it = 0; it < NI; ++it) {
            const int idx = g + it * T;
            if (idx >= 6 * NF) continue;
            for (int d = 0; d < 3; ++d) sL[(idx / NF * 3 + d) * NF + idx % NF] = c_of(c_d(sN[d * 6 * NF + idx]) * face[it]);
          }
          col_sync<N>(grp);
          if (act)
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              double s = 0.0;
              for (int a = 0; a < 3; ++a) {
                const int st = a == 0 ? 1 : a == 1 ? N : N * N;
                const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
                for (int side = 0; side < 2; ++side)
                  s = fma(so.deh[side][i], c_d(sL[((2 * a + side) * 3 + d) * NF + fp]), s);
                for (int k = 0; k < N; ++k) s = fma(-so.dDh[k * N + i], c_d(sY[(a * 3 + d) * NP + base + k * st]), s);
              }
              q[d] = s * gue[10 * NP + g];
              sQ[d * NP + g] = c_of(q[d]);
            }
          col_sync<N>(grp);
#pragma unroll
          for (int it = 0; it < NI; ++it) {
            const int idx = g + it * T;
            if (idx >= 6 * NF) continue;
#pragma unroll
            for (int d = 0; d < 3; ++d) {
              double s = 0.0;
              for (int k = 0; k < N; ++k) s = fma(so.de[(idx / NF) & 1][k], c_d(sQ[d * NP + tb[it] + k * ts[it]]), s);
              qtr[it][d] = s;
            }
          }
        }
      };
      gradient(ud, hat, qd, qt);
      if (c == 0 && has_wall) {              // varrho moves the wall's energy trace
#pragma unroll
        for (int it = 0; it < NI; ++it) hat[it] = g + it * T < 6 * NF ? uw[g + it * T] * uft[it] : 0.0;
        // (|uw| may exceed the range of a unit value: scaled by a power of two, linear in it)
        double top = 0.0;
        for (int k = 0; k < 6 * NF; ++k) top = fmax(top, fabs(uw[k]));
        int ex = 0;
        frexp(top, &ex);
#pragma unroll
        for (int it = 0; it < NI; ++it) hat[it] = ldexp(hat[it], -ex);
        gradient(0.0, hat, qw, qwt);
#pragma unroll
        for (int d = 0; d < 3; ++d) qw[d] = ldexp(qw[d], ex);
#pragma unroll
        for (int it = 0; it < NI; ++it)
#pragma unroll
          for (int d = 0; d < 3; ++d) qwt[it][d] = ldexp(qwt[it][d], ex);
      }
      // pointwise Jacobians
      double F[20];
      int mx[5] = {0, 0, 0, 0, 0};
      if (act) {
#pragma unroll
        for (int r = 0; r < 20; ++r) {
          const double* A = VA + r * NP + g;
          F[r] = fma(A[0], ud, fma(A[20 * NP], qd[0], fma(A[40 * NP], qd[1], A[60 * NP] * qd[2])));
        }
        if (c == 0 && has_wall)
#pragma unroll
          for (int r = 0; r < 20; ++r)
#pragma unroll
            for (int d = 0; d < 3; ++d) F[r] = fma(JV[((eb * 20 + 9 + 5 * d) * 20 + r) * NP + g], qw[d], F[r]);
        const double w = -det * inv_c * ud;  // J_G = -c (J_r - M / c)
#pragma unroll
        for (int k = 0; k < 5; ++k) F[15 + k] += k == c ? w : 0.0;
#pragma unroll
        for (int r = 0; r < 20; ++r) mx[r % 5] = max(mx[r % 5], fx_mag(F[r]));
      }
      col_sync<N>(grp);                      // the gradient's cells have been read
      if (act)
#pragma unroll
        for (int r = 0; r < 15; ++r) sF[r * NP + g] = c_of(F[r]);
#pragma unroll
      for (int it = 0; it < NI; ++it) {
        const int idx = g + it * T;
        if (idx >= 6 * NF) continue;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const double* A = FA + k * 6 * NF + idx;
          double h = fma(A[0], uft[it], fma(A[30 * NF], qt[it][0], fma(A[60 * NF], qt[it][1], A[90 * NF] * qt[it][2])));
          if (c == 0 && has_wall)
#pragma unroll
            for (int d = 0; d < 3; ++d) h = fma(JF[((eb * 20 + 9 + 5 * d) * 5 + k) * 6 * NF + idx], qwt[it][d], h);
          sH[k * 6 * NF + idx] = c_of(h);
          mx[k] = max(mx[k], fx_mag(h));
        }
      }
      col_max<N, 5>(mx, red, grp);
      bool ok = true;
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        ok = ok && fx_ok(mx[k]);
        mx[k] = fx_exp(mx[k]);
      }
      if constexpr (T < 32) ok = __all_sync(0xffffffffu, ok);
      cell *b0 = sF, *b1 = sF + 5 * NP;
      float col[5];
      if (ok) {
        if (act)
#pragma unroll
          for (int r = 0; r < 15; ++r) sF[r * NP + g] = c_split<28>(fx_from<58>(F[r], mx[r % 5]));
#pragma unroll
        for (int it = 0; it < NI; ++it) {
          const int idx = g + it * T;
          if (idx >= 6 * NF) continue;
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            cell& x = sH[k * 6 * NF + idx];
            x = c_split<28>(fx_from<58>(c_d(x), mx[k]));
          }
        }
        col_sync<N>(grp);
        long long R[5] = {0, 0, 0, 0, 0};
        int up[5];
        if (act) {
          fxacc s[5] = {fx_zero<28>(), fx_zero<28>(), fx_zero<28>(), fx_zero<28>(), fx_zero<28>()};
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            const int st = a == 0 ? 1 : a == 1 ? N : N * N;
            const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
#pragma unroll
            for (int side = 0; side < 2; ++side) {
              const fx ev = c_fx(so.lift[side][i]);
#pragma unroll
              for (int k = 0; k < 5; ++k) fx_mac(s[k], ev, c_fx(sH[k * 6 * NF + (2 * a + side) * NF + fp]));
            }
#pragma unroll
            for (int q = 0; q < N; ++q) {
              const fx D = c_fx(so.Dn[q * N + i]);
#pragma unroll
              for (int k = 0; k < 5; ++k) fx_mac(s[k], D, c_fx(sF[(a * 5 + k) * NP + base + q * st]));
            }
          }
#pragma unroll
          for (int k = 0; k < 5; ++k) R[k] = ((fx_from<58>(F[15 + k], mx[k]) + 1) >> 1) - fx_sum<28>(s[k]);
        }
#pragma unroll
        for (int k = 0; k < 5; ++k) up[k] = (int)((R[k] < 0 ? -R[k] : R[k]) >> 32);
        col_sync<N>(grp);
        col_max<N, 5>(up, red, grp);
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          up[k] = up[k] < (1 << 26) ? 0 : 6 - __clz(up[k]);
          if (act) b0[k * NP + g] = c_split<30>(R[k] >> up[k]);
        }
        col_sync<N>(grp);
        if (act) pass_b<N, 0, true, true, 5>(so, b0, b1, g);
        col_sync<N>(grp);
        if (act) pass_b<N, 1, true, true, 5>(so, b1, b0, g);
        col_sync<N>(grp);
        if (act) {
          pass_b<N, 2, true, true, 5>(so, b0, b1, g);
#pragma unroll
          for (int k = 0; k < 5; ++k)
            col[k] = (float)(-stage_c * fx_to_double(fx_join<30>(c_fx(b1[k * NP + g])), mx[k] - 1079 + up[k]));
        }
      } else {                               // FP64 twin
        col_sync<N>(grp);
        double R[5];
        if (act)
          for (int k = 0; k < 5; ++k) {
            double s = F[15 + k];
            for (int a = 0; a < 3; ++a) {
              const int st = a == 0 ? 1 : a == 1 ? N : N * N;
              const int i = ig[a], base = g - i * st, fp = vol_face_point<N>(g, a);
              for (int q = 0; q < N; ++q) s = fma(so.dDh[q * N + i], c_d(sF[(a * 5 + k) * NP + base + q * st]), s);
              for (int side = 0; side < 2; ++side) s = fma(-so.deh[side][i], c_d(sH[k * 6 * NF + (2 * a + side) * NF + fp]), s);
            }
            R[k] = s;
          }
        col_sync<N>(grp);
        if (act)
          for (int k = 0; k < 5; ++k) b0[k * NP + g] = c_of(R[k]);
        col_sync<N>(grp);
        if (act) pass_b<N, 0, true, false, 5>(so, b0, b1, g);
        col_sync<N>(grp);
        if (act) pass_b<N, 1, true, false, 5>(so, b1, b0, g);
        col_sync<N>(grp);
        if (act) {
          pass_b<N, 2, true, false, 5>(so, b0, b1, g);
          for (int k = 0; k < 5; ++k) col[k] = (float)(-stage_c * c_d(b1[k * NP + g]));
        }
      }
      if (act && live)
#pragma unroll
        for (int k = 0; k < 5; ++k) out[(e * n + c * NP + b) * (long long)n + k * NP + g] = col[k];
    }
  }
}

// --------------------------------------------------------------------------------------------
// FP32 assembly, for steps whose inner operator is the FP32 one (jv_prec f32)
// --------------------------------------------------------------------------------------------
// The same columns from FP32 Jacobians, geometry and sums (the weighted geometry of the FP32 kernels). The
// gradient of a unit value needs no contraction through shared memory: its line values are products of entries
// of B, so a thread keeps D G / (w |J|) of its lines and e n / (w |J|) of its faces in registers for all columns.
// In FP64 the assembly is bound by the FP64 pipe and by the fixed point's issue; here by issue and shared-memory loads.
// Set-up (assembly, inversion, FP16 copies) of 98,304 degree-2 blocks 309 ms in FP64, 245 with FP32 probing of the
// tangent, 99 now (43 of it assembly); of 24,576 degree-3 blocks 365 in FP64, 322 with probing, 147 now.
template <int N>
struct Blk32 {
  static constexpr int NP = N * N * N, NF = N * N;
  static constexpr int T = Blk<N>::T, GP = Blk<N>::GP;
  // floats of a column: gradient [3][NP], then reference fluxes [15][NP], then the passes; face fluxes [5][6 NF];
  // traces of the column's variable [6 NF]
  static constexpr int W = 15 * NP + 36 * NF;
  static constexpr int floats = 80 * NP + 120 * NF + GP * W;
};

template <int N>
__global__ void __launch_bounds__(128) k_jac_volume32(long long e0, long long nE, PhysT<float> P, float t,
                                                      const float* __restrict__ geo, const float* __restrict__ accg,
                                                      const float* __restrict__ xg, const float* __restrict__ ug,
                                                      const float* __restrict__ qg, const float* __restrict__ mixg,
                                                      float* __restrict__ JV) {
  using D32 = DualT<float>;
  constexpr int NP = Blk32<N>::NP;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nE * NP) return;
  const long long eb = i / NP, e = e0 + eb;
  const int g = (int)(i % NP);
  float x3[3] = {0.f, 0.f, 0.f}, mg[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, G[9];
  const float a3[3] = {accg[e * 3 * NP + g], accg[e * 3 * NP + NP + g], accg[e * 3 * NP + 2 * NP + g]};
  if (P.euv)
    for (int d = 0; d < 3; ++d) x3[d] = xg[e * 3 * NP + d * NP + g];
  if (P.comp)
    for (int k = 0; k < 8; ++k) mg[k] = mixg[(e * 8 + k) * NP + g];
  const float* gp = geo + e * 10 * NP + g;
#pragma unroll
  for (int k = 0; k < 9; ++k) G[k] = gp[k * NP];
  const float Wd = gp[9 * NP];
#pragma unroll 1
  for (int dir = 0; dir < 20; ++dir) {
    D32 u[5], q[3][5], F[3][5], src[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) u[c] = D32{ug[(e * 5 + c) * NP + g], dir == c ? 1.f : 0.f};
#pragma unroll
    for (int k = 0; k < 15; ++k) q[k / 5][k % 5] = D32{qg[(e * 15 + k) * NP + g], dir == 5 + k ? 1.f : 0.f};
    volume_point<D32>(P, u, q, G, Wd, a3, x3, t, F, src, mg);
    float* out = JV + (eb * 20 + dir) * 20 * NP + g;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int c = 0; c < 5; ++c) out[(a * 5 + c) * NP] = F[a][c].d;
#pragma unroll
    for (int c = 0; c < 5; ++c) out[(15 + c) * NP] = src[c].d;
  }
}

template <int N>
__global__ void __launch_bounds__(128) k_jac_faces32(long long e0, long long nE, PhysT<float> P,
                                                     const int* __restrict__ nbr, const int* __restrict__ nbr_fo,
                                                     const float* __restrict__ fgeo, const double* __restrict__ kn,
                                                     const float* __restrict__ uf, const float* __restrict__ qf,
                                                     const float* __restrict__ mixf, float* __restrict__ JF) {
  using D32 = DualT<float>;
  constexpr int NF = Blk32<N>::NF;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nE * 6 * NF) return;
  const long long eb = i / (6 * NF), e = e0 + eb;
  const int phi = (int)(i / NF % 6), f = (int)(i % NF);
  const long long face = e * 6 + phi;
  const int nb = nbr[face];
  Mix<float> mx{P.cv, 1.f};
  if (P.comp) {
    mx.cv = mixf[(face * 2) * NF + f];
    mx.kfac = mixf[(face * 2 + 1) * NF + f];
  }
  const float* gp = fgeo + face * 4 * NF + f;
  const float n[3] = {gp[0], gp[NF], gp[2 * NF]}, area = gp[3 * NF];
  long long face2 = face;
  int f2 = f;
  if (nb >= 0) {
    const int fo = nbr_fo[face];
    face2 = (long long)nb * 6 + (fo & 7);
    f2 = orient_map(fo >> 3, f % N, f / N, N);
  }
  const float kn2[3] = {(float)kn[face2 * 3 * NF + f2], (float)kn[(face2 * 3 + 1) * NF + f2],
                        (float)kn[(face2 * 3 + 2) * NF + f2]};
  float* out = JF + eb * 600 * NF + phi * NF + f;
#pragma unroll 1
  for (int dir = 0; dir < 20; ++dir) {
    D32 u[5], q[3][5], res[5];
#pragma unroll
    for (int c = 0; c < 5; ++c) u[c] = D32{uf[(face * 5 + c) * NF + f], dir == c ? 1.f : 0.f};
#pragma unroll
    for (int k = 0; k < 15; ++k) q[k / 5][k % 5] = D32{qf[(face * 15 + k) * NF + f], dir == 5 + k ? 1.f : 0.f};
    if (nb >= 0) {
      // the other side answers through its gradient alone
      D32 u2[5], q2[3][5];
#pragma unroll
      for (int c = 0; c < 5; ++c) u2[c] = D32{uf[(face2 * 5 + c) * NF + f2], 0.f};
#pragma unroll
      for (int k = 0; k < 15; ++k) q2[k / 5][k % 5] = D32{qf[(face2 * 15 + k) * NF + f2], k % 5 == dir ? kn2[k / 5] : 0.f};
      face_flux_interior(P, u, q, u2, q2, n, area, res, mx);
    } else if (nb == -DG_BC_WALL) {
      D32 ub[5], sg[5];
      wall_trace(P, u, ub);
      flux_dot_n(P, ub, q, n, true, res, mx);
      sigma_diag(P, ub, sg, mx);
#pragma unroll
      for (int c = 0; c < 5; ++c) res[c] = res[c] + sg[c] * (area * (u[c] - ub[c]));
    } else {
      flux_dot_n(P, u, q, n, false, res, mx);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) out[(dir * 5 + k) * 6 * NF] = res[k].d;
  }
}

template <int N>
__global__ void __launch_bounds__(Blk32<N>::GP * Blk32<N>::T, 2)
    k_blocks32(long long e0, const Ops* __restrict__ ops, float t_wall, const float* __restrict__ geo,
               const float* __restrict__ fgeo, const int* __restrict__ nbr, const float* __restrict__ uf,
               const float* __restrict__ JV, const float* __restrict__ JF, float stage_c, float* __restrict__ out) {
  using B = Blk32<N>;
  constexpr int NP = B::NP, NF = B::NF, T = B::T, GP = B::GP, NI = Grp<N>::NI, n = 5 * NP;
  __shared__ SmemOpsT<float> so;
  __shared__ float uw[6 * NF];               // d u_hat_4 / d varrho at wall face points, else 0
  extern __shared__ __align__(16) float sm32[];
  load_ops<N, float>(ops, so);
  const int grp = threadIdx.x / T, g = threadIdx.x % T;
  const bool act = g < NP;
  const long long eb = blockIdx.x, e = e0 + eb;
  float* VA = sm32;                          // [4][20][NP] Jacobian columns u_c, q_0c, q_1c, q_2c
  float* FA = VA + 80 * NP;                  // [4][5][6 NF]
  float* sF = FA + 120 * NF + grp * B::W;    // [15][NP]
  float* sH = sF + 15 * NP;                  // [5][6 NF]
  float* sT = sH + 30 * NF;                  // [6 NF]
  bool has_wall = false;
  for (int phi = 0; phi < 6; ++phi) has_wall = has_wall || nbr[e * 6 + phi] == -DG_BC_WALL;
  for (int i = threadIdx.x; i < 6 * NF; i += blockDim.x)
    uw[i] = nbr[e * 6 + i / NF] == -DG_BC_WALL ? 0.5f * t_wall * expf(0.5f * uf[(e * 6 + i / NF) * 5 * NF + i % NF]) : 0.f;
  __syncthreads();
  const int ig[3] = {g % N, (g / N) % N, g / (N * N) % N};
  int fp[3], lb[3];
  float DG[3][N][3], en[6][3], D[3][N], ec[6], Wd = 0.f;
  axis_coefs<N, true>(so.D, ig, D);
  end_coefs(so, ig, ec);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lb[a] = g - ig[a] * pt_stride<N>(a);
    fp[a] = vol_face_point<N>(g, a);
  }
  if (act) {
    const float* gp = geo + e * 10 * NP;
    Wd = gp[9 * NP + g];
    const float iW = 1.f / Wd;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int k = 0; k < N; ++k) DG[a][k][d] = -D[a][k] * gp[(a * 3 + d) * NP + lb[a] + k * pt_stride<N>(a)] * iW;
#pragma unroll
        for (int side = 0; side < 2; ++side)
          en[2 * a + side][d] = ec[2 * a + side] * fgeo[((e * 6 + 2 * a + side) * 4 + d) * NF + fp[a]] * iW;
      }
  }
  int tb[NI], ts[NI];
#pragma unroll
  for (int it = 0; it < NI; ++it) face_line<N>((g + it * T) / NF, (g + it * T) % NF, tb[it], ts[it]);
#pragma unroll 1
  for (int c = 0; c < 5; ++c) {
    __syncthreads();
    for (int i = threadIdx.x; i < 80 * NP; i += blockDim.x) {
      const int k = i / (20 * NP);
      VA[i] = JV[(eb * 20 + (k ? 5 * k + c : c)) * 20 * NP + i % (20 * NP)];
    }
    for (int i = threadIdx.x; i < 120 * NF; i += blockDim.x) {
      const int k = i / (30 * NF);
      FA[i] = JF[(eb * 20 + (k ? 5 * k + c : c)) * 30 * NF + i % (30 * NF)];
    }
    __syncthreads();
    for (int b = grp; b < (NP + GP - 1) / GP * GP; b += GP) {
      // (every group runs the same number of columns; those beyond the last one write nothing)
      const int ib[3] = {b % N, (b / N) % N, b / (N * N) % N};
      const float Bo[3] = {so.B[ig[0] * N + ib[0]], so.B[ig[1] * N + ib[1]], so.B[ig[2] * N + ib[2]]};
      const float ud = Bo[0] * Bo[1] * Bo[2];
      float uft[NI], qt[NI][3], qw[3] = {0.f, 0.f, 0.f}, qwt[NI][3];
      // gradient of the traces in sT and, when vol, of the unit value; and its face traces
      auto gradient = [&](bool vol, float (&q)[3], float (&qtr)[NI][3]) {
        col_sync<N>(grp);
        if (act) {
#pragma unroll
          for (int d = 0; d < 3; ++d) q[d] = 0.f;
#pragma unroll
          for (int phi = 0; phi < 6; ++phi) {
            const float x = sT[phi * NF + fp[phi >> 1]];
#pragma unroll
            for (int d = 0; d < 3; ++d) q[d] = fmaf(en[phi][d], x, q[d]);
          }
          if (vol)
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              const float rest = Bo[(a + 1) % 3] * Bo[(a + 2) % 3];
#pragma unroll
              for (int k = 0; k < N; ++k) {
                const float x = so.B[k * N + ib[a]] * rest;
#pragma unroll
                for (int d = 0; d < 3; ++d) q[d] = fmaf(DG[a][k][d], x, q[d]);
              }
            }
#pragma unroll
          for (int d = 0; d < 3; ++d) sF[d * NP + g] = q[d];
        }
        col_sync<N>(grp);
#pragma unroll
        for (int it = 0; it < NI; ++it) {
          const int idx = g + it * T;
          if (idx >= 6 * NF) continue;
          const float* ev = ((idx / NF) & 1) ? so.eR : so.eL;
#pragma unroll
          for (int d = 0; d < 3; ++d) {
            qtr[it][d] = 0.f;
#pragma unroll
            for (int k = 0; k < N; ++k) qtr[it][d] = fmaf(ev[k], sF[d * NP + tb[it] + k * ts[it]], qtr[it][d]);
          }
        }
        col_sync<N>(grp);
      };
      // its traces: l_b(-1), l_b(1) are 1 at the end nodes, else 0
#pragma unroll
      for (int it = 0; it < NI; ++it) {
        const int idx = g + it * T, phi = idx / NF, f = idx % NF, axis = phi >> 1;
        uft[it] = 0.f;
        if (idx >= 6 * NF) continue;
        const int s_ax = axis == 0 ? 1 : 0, t_ax = axis == 2 ? 1 : 2;
        if (ib[axis] == ((phi & 1) ? N - 1 : 0)) uft[it] = so.B[f % N * N + ib[s_ax]] * so.B[f / N * N + ib[t_ax]];
        const int nb = nbr[e * 6 + phi];
        sT[idx] = nb >= 0 ? 0.5f * uft[it] : nb == -DG_BC_OUTFLOW ? uft[it] : c == 0 ? uft[it] : 0.f;
      }
      float qd[3] = {0.f, 0.f, 0.f};
      gradient(true, qd, qt);
      if (c == 0 && has_wall) {              // varrho moves the wall's energy trace
#pragma unroll
        for (int it = 0; it < NI; ++it)
          if (g + it * T < 6 * NF) sT[g + it * T] = uw[g + it * T] * uft[it];
        gradient(false, qw, qwt);
      }
      float src[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (act)
#pragma unroll
        for (int r = 0; r < 20; ++r) {
          const float* A = VA + r * NP + g;
          float x = fmaf(A[0], ud, fmaf(A[20 * NP], qd[0], fmaf(A[40 * NP], qd[1], A[60 * NP] * qd[2])));
          if (c == 0 && has_wall)
#pragma unroll
            for (int d = 0; d < 3; ++d) x = fmaf(JV[((eb * 20 + 9 + 5 * d) * 20 + r) * NP + g], qw[d], x);
          if (r < 15) sF[r * NP + g] = x;
          else src[r - 15] = x;
        }
#pragma unroll
      for (int it = 0; it < NI; ++it) {
        const int idx = g + it * T;
        if (idx >= 6 * NF) continue;
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          const float* A = FA + k * 6 * NF + idx;
          float h = fmaf(A[0], uft[it], fmaf(A[30 * NF], qt[it][0], fmaf(A[60 * NF], qt[it][1], A[90 * NF] * qt[it][2])));
          if (c == 0 && has_wall)
#pragma unroll
            for (int d = 0; d < 3; ++d) h = fmaf(JF[((eb * 20 + 9 + 5 * d) * 5 + k) * 6 * NF + idx], qwt[it][d], h);
          sH[k * 6 * NF + idx] = h;
        }
      }
      col_sync<N>(grp);
      float R[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
      if (act)
#pragma unroll
        for (int k = 0; k < 5; ++k) {
          float x = src[k];
#pragma unroll
          for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int q = 0; q < N; ++q) x = fmaf(D[a][q], sF[(a * 5 + k) * NP + lb[a] + q * pt_stride<N>(a)], x);
#pragma unroll
          for (int phi = 0; phi < 6; ++phi) x = fmaf(-ec[phi], sH[k * 6 * NF + phi * NF + fp[phi >> 1]], x);
          R[k] = (k == c ? Wd * ud : 0.f) - stage_c * x;
        }
      col_sync<N>(grp);
      // B^T along each direction
      float *in = sF, *to = sF + 5 * NP;
      if (act)
#pragma unroll
        for (int k = 0; k < 5; ++k) in[k * NP + g] = R[k];
      col_sync<N>(grp);
#pragma unroll
      for (int dir = 0; dir < 3; ++dir) {
        if (act)
#pragma unroll
          for (int k = 0; k < 5; ++k) {
            float x = 0.f;
#pragma unroll
            for (int q = 0; q < N; ++q) x = fmaf(so.B[q * N + ig[dir]], in[k * NP + lb[dir] + q * pt_stride<N>(dir)], x);
            if (dir < 2) to[k * NP + g] = x;
            else if (b < NP) out[(e * n + c * NP + b) * (long long)n + k * NP + g] = x;
          }
        col_sync<N>(grp);
        float* z = in;
        in = to;
        to = z;
      }
    }
  }
}

}  // namespace dg
