// FP64 element and face kernels of the LDG residual, its exact tangent and the mass matrix.
//
// Representation. A degree-p field on an element is held by its values at the (p+1)^3 Gauss
// points ("Gauss space"). The ABI's nodal GLL coefficients map to Gauss space by B x B x B, with
// B[q][a] = l^GLL_a(eta_q) invertible. In Gauss space the operators of Eq. DGformulation reduce
// to exact sum-factorised 1D passes:
//   derivative along xi_a ............ D (Lagrange derivative on the Gauss points)
//   value on face xi_a = -1 / +1 ...... eL / eR (Lagrange extrapolation to the end points)
//   test-function weak derivative .... D^T;  face lifting ... eL / eR outer products
// and the element mass matrix is M = B^T W B with W = diag(w_g |J_g|), so
//   Gradient (Eq. DGformulation a):  Q_{d,c} = W^{-1} [ -sum_a D_a^T (G_{a d} U_c)
//                                                       + sum_faces e_face (w n_d dS) U_hat_c ]
//   Residual (Eq. DGformulation b):  r = B^T [ sum_a D_a^T (sum_d G_{a d} F_{c d}) + W s_c
//                                              - sum_faces e_face (F_hat . w n dS)_c ]
// with G_{a d} = w_g |J| d xi_a / d x_d (cofactor of the Jacobian). Each identity is exact
// (p-degree polynomials, the same quadrature), so these kernels compute the same discrete
// operator as a dense nodal implementation, up to rounding.
//
// Kernels (one CTA handles EPB elements, one thread per Gauss point; faces one thread per point). The
// kernels of this file named k_interp, k_grad and k_volume are the FP32 ones; their FP64 counterparts
// k_interp64, k_grad64 and k_volume64 (dg_fp64.cuh) run the contractions in block fixed point.
//   k_interp   nodal u (and tangent v) -> Gauss values U, face traces UF
//   k_grad     U, UF (own + neighbour) -> Q in Gauss space, face traces QF
//   k_faces    UF, QF of both sides -> F_hat . (w n dS) for both element faces (Eq. LDG2)
//   k_volume   U, Q, F_hat -> pointwise F, s; projection; lifting; B^T -> nodal r (and J v)
// The exact Jacobian-vector product carries forward-mode dual numbers through every step.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <string>
#include <type_traits>

#include "dg_bits.cuh"
#include "dg_internal.cuh"
#include "dg_phys64.cuh"

namespace dg {

template <int N>
struct Shape {
  static constexpr int NP = N * N * N;
  static constexpr int NF = N * N;
};

// elements per CTA by kernel footprint
template <int N, int NC>
struct Epb {
  static constexpr int value = (N == 2) ? 16 : (N == 3) ? 8 : (N == 4) ? (NC == 1 ? 4 : 2) : (NC == 1 ? 2 : 1);
};

template <int N>
__device__ __forceinline__ int pt_stride(int dir) {
  return dir == 0 ? 1 : (dir == 1 ? N : N * N);
}

// Contraction modes of the basis operators (the FP32 path only): CM_NATIVE multiplies in the
// working precision; CM_BF16 / CM_FP16 round both operands to bfloat16 / binary16 and accumulate
// in FP32 (the products of two such values are exact in FP32, as in a tensor-core MMA);
// CM_BF16X3 / CM_FP16X3 split each operand into hi + lo parts and keep three of the four products
// (hi*hi + hi*lo + lo*hi).
enum { CM_NATIVE = 0, CM_BF16 = 1, CM_FP16 = 2, CM_BF16X3 = 3, CM_FP16X3 = 4 };

template <int CM> __device__ __forceinline__ float cm_round(float v);
template <> __device__ __forceinline__ float cm_round<CM_BF16>(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }
template <> __device__ __forceinline__ float cm_round<CM_FP16>(float v) { return __half2float(__float2half_rn(v)); }

template <int CM, typename R>
__device__ __forceinline__ R cm_fma(R a, R x, R acc) {
  if constexpr (CM == CM_NATIVE) {
    return fma(a, x, acc);
  } else {
    constexpr int B = (CM == CM_BF16 || CM == CM_BF16X3) ? CM_BF16 : CM_FP16;
    const float ah = cm_round<B>(a), xh = cm_round<B>(x);
    if constexpr (CM == CM_BF16 || CM == CM_FP16) {
      return fmaf(ah, xh, acc);
    } else {
      const float al = cm_round<B>(a - ah), xl = cm_round<B>(x - xh);
      return fmaf(ah, xh, fmaf(ah, xl, fmaf(al, xh, acc)));
    }
  }
}

// 1D pass along `dir` at point g: sum_k A[i][k] in[.. k ..] (T = false) or A[k][i] (T = true)
template <int N, bool T, typename R, int CM = CM_NATIVE>
__device__ __forceinline__ R line(const R* __restrict__ A, const R* __restrict__ in, int g, int dir) {
  const int st = pt_stride<N>(dir);
  const int i = (g / st) % N;
  const int base = g - i * st;
  R acc = R(0);
#pragma unroll
  for (int k = 0; k < N; ++k) acc = cm_fma<CM>(T ? A[k * N + i] : A[i * N + k], in[base + k * st], acc);
  return acc;
}

// Gauss point index of (face phi, face point f, index k along the face normal)
template <int N>
__device__ __forceinline__ int face_vol_point(int phi, int f, int k) {
  const int axis = phi >> 1;
  const int is = f % N, it = f / N;
  int i0, i1, i2;
  if (axis == 0) { i0 = k; i1 = is; i2 = it; }
  else if (axis == 1) { i0 = is; i1 = k; i2 = it; }
  else { i0 = is; i1 = it; i2 = k; }
  return i0 + N * (i1 + N * i2);
}

// face point of volume point g on a face of the given axis
template <int N>
__device__ __forceinline__ int vol_face_point(int g, int axis) {
  const int i0 = g % N, i1 = (g / N) % N, i2 = g / (N * N);
  if (axis == 0) return i1 + N * i2;
  if (axis == 1) return i0 + N * i2;
  return i0 + N * i1;
}

template <typename R>
struct SmemOpsT {
  R B[MAXN * MAXN], D[MAXN * MAXN], Binv[MAXN * MAXN], eL[MAXN], eR[MAXN];
};
using SmemOps = SmemOpsT<double>;

// the 1D operators (built in FP64 on the host) rounded to the working precision
template <int N, typename R>
__device__ __forceinline__ void load_ops(const Ops* __restrict__ o, SmemOpsT<R>& s) {
  for (int i = threadIdx.x; i < N * N; i += blockDim.x) {
    s.B[i] = (R)o->B[i];
    s.D[i] = (R)o->D[i];
    s.Binv[i] = (R)o->Binv[i];
  }
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    s.eL[i] = (R)o->eL[i];
    s.eR[i] = (R)o->eR[i];
  }
}


// NC values of one entry (value and tangent planes), moved through shared memory by one access
template <int V, typename R>
struct alignas(V * sizeof(R)) Pack { R v[V]; };

// the 1D operator entries of this thread's point, held in registers: along each axis the column i of A
// (T: sum over k of A[k][i] x_k), else its row
template <int N, bool T, typename R>
__device__ __forceinline__ void axis_coefs(const R* A, const int (&ig)[3], R (&out)[3][N]) {
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int k = 0; k < N; ++k) out[a][k] = T ? A[k * N + ig[a]] : A[ig[a] * N + k];
}
// the two end-point coefficients of this thread's point along each axis, in face order
template <typename R>
__device__ __forceinline__ void end_coefs(const SmemOpsT<R>& so, const int (&ig)[3], R (&out)[6]) {
#pragma unroll
  for (int phi = 0; phi < 6; ++phi) out[phi] = ((phi & 1) ? so.eR : so.eL)[ig[phi >> 1]];
}

// the extrapolations of a line of N entries to its two ends
template <int N, int CM, int V, typename R>
__device__ __forceinline__ void line_ends(const SmemOpsT<R>& so, const Pack<V, R>* in, int st, Pack<V, R> (&end)[2]) {
#pragma unroll
  for (int p = 0; p < V; ++p) end[0].v[p] = end[1].v[p] = R(0);
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const Pack<V, R> x = in[k * st];
#pragma unroll
    for (int p = 0; p < V; ++p) {
      end[0].v[p] = cm_fma<CM>(so.eL[k], x.v[p], end[0].v[p]);
      end[1].v[p] = cm_fma<CM>(so.eR[k], x.v[p], end[1].v[p]);
    }
  }
}

// FP64 <-> FP32 at the nodal ends of the FP32 path: the integer conversions, since a cvt issues on the FP64
// pipe (2 per cycle and SM)
// (one branch for K values, after all of them have been loaded)
static __device__ __noinline__ float cvt_any(double x) { return (float)x; }
template <int K, typename R>
__device__ __forceinline__ void from_f64(const double (&x)[K], R (&y)[K]) {
  if constexpr (std::is_same<R, float>::value) {
    bool plain = true;
#pragma unroll
    for (int k = 0; k < K; ++k) plain = plain && to_f32_plain(x[k]);
    if (plain) {
#pragma unroll
      for (int k = 0; k < K; ++k) y[k] = to_f32_rn(x[k]);
    } else {
#pragma unroll
      for (int k = 0; k < K; ++k) y[k] = cvt_any(x[k]);
    }
  } else {
#pragma unroll
    for (int k = 0; k < K; ++k) y[k] = (R)x[k];
  }
}
template <typename R>
__device__ __forceinline__ double as_f64(R x) {
  if constexpr (std::is_same<R, float>::value) return to_f64_exact(x);
  else return (double)x;
}

// The element kernels below give each thread one Gauss point and pass lines through shared memory. They were
// bound by instruction issue and the load/store unit, most of it not the contraction: operator entries read
// again for every variable, index arithmetic, FP64 conversions. Operator entries and line addresses now stay
// in registers, value and tangent go through shared memory as one 8-byte entry, results leave from registers,
// and conversions run on the integer pipe; every sum keeps its order. Jv and r of 27,648 degree-3 elements:
//   k_interp 81 -> 74 us (shared-memory bandwidth), k_grad 321 -> 232, k_volume 268 -> 188; k_faces 101
//   (DRAM); HBM traffic alone 47, 135, 81 and 85.

// --------------------------------------------------------------------------------------------
// k_interp: nodal -> Gauss values and face traces. NC = 1 (u) or 2 (u and tangent v).
// --------------------------------------------------------------------------------------------
template <int N, int NC, typename R, int CM = CM_NATIVE>
__global__ void __launch_bounds__(Epb<N, NC>::value * Shape<N>::NP)
    k_interp(const double* __restrict__ u, const double* __restrict__ v, long long E,
             const Ops* __restrict__ ops, R* __restrict__ ug, R* __restrict__ uf) {
  constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF, EPB = Epb<N, NC>::value, NT = EPB * NP;
  using V = Pack<NC, R>;
  __shared__ SmemOpsT<R> so;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* b0 = reinterpret_cast<V*>(smem_raw);   // [5][NT]
  V* b1 = b0 + 5 * NT;                      // [5][NT]
  load_ops<N, R>(ops, so);
  const int tid = threadIdx.x, g = tid % NP;
  const long long e0 = (long long)blockIdx.x * EPB, e = e0 + tid / NP;
  const bool active = e < E;
  if (active) {
    double x[5 * NC];
#pragma unroll
    for (int c = 0; c < 5 * NC; ++c) x[c] = (c < 5 ? u : v)[e * 5 * NP + c % 5 * NP + g];
    R y[5 * NC];
    from_f64<5 * NC>(x, y);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      V z;
#pragma unroll
      for (int p = 0; p < NC; ++p) z.v[p] = y[p * 5 + c];
      b0[c * NT + tid] = z;
    }
  }
  __syncthreads();
  const long long plane_g = E * 5 * NP;
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  V *in = b0, *out = b1;
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const int st = pt_stride<N>(dir), base = tid - ig[dir] * st;
    R B[N];
#pragma unroll
    for (int k = 0; k < N; ++k) B[k] = so.B[ig[dir] * N + k];
    if (active)
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        V acc;
#pragma unroll
        for (int p = 0; p < NC; ++p) acc.v[p] = R(0);
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const V x = in[c * NT + base + k * st];
#pragma unroll
          for (int p = 0; p < NC; ++p) acc.v[p] = cm_fma<CM>(B[k], x.v[p], acc.v[p]);
        }
        out[c * NT + tid] = acc;
        if (dir == 2)
#pragma unroll
          for (int p = 0; p < NC; ++p) ug[p * plane_g + e * 5 * NP + c * NP + g] = acc.v[p];
      }
    __syncthreads();
    V* t = in;
    in = out;
    out = t;
  }
  // `in` holds Gauss values; face traces, both ends of a line per iteration
  const long long plane_f = E * 6 * 5 * NF;
  for (int idx = tid; idx < EPB * 3 * NF; idx += NT) {
    const int l = idx / (3 * NF), a = (idx / NF) % 3, f = idx % NF;
    if (e0 + l >= E) continue;
    const int base = l * NP + face_vol_point<N>(2 * a, f, 0), st = pt_stride<N>(a);
    R* dst = uf + (e0 + l) * 30 * NF + a * 10 * NF + f;
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      V end[2];
      line_ends<N, CM>(so, in + c * NT + base, st, end);
#pragma unroll
      for (int side = 0; side < 2; ++side)
#pragma unroll
        for (int p = 0; p < NC; ++p) dst[p * plane_f + (side * 5 + c) * NF] = end[side].v[p];
    }
  }
}

// --------------------------------------------------------------------------------------------
// k_grad: LDG gradient in Gauss space (Eq. DGformulation a) and its face traces
// --------------------------------------------------------------------------------------------
// Shared memory holds the field and its traces alone: a line's products G u and a face's n u_hat are formed
// again by every point that adds them, from geometry that stays in registers for all variables (N + 2 entries
// per axis). That takes 3 FP32 multiplications for each shared load it saves; storing the products made shared-
// memory bandwidth the bound (289 us). 4 CTAs per SM at 128 registers; more CTAs with fewer registers are
// slower (236, 252).
// TO (tangent only, NC = 1): the value plane of ug, uf, qg, qf already holds the state's values
// (computed once for all the Jv of one Krylov solve);
// only the tangent plane is formed, with the same arithmetic as the tangent of NC = 2, so the
// result is identical. The wall trace of the tangent reads the value plane's varrho trace.
template <int N, int NC, typename R, int CM = CM_NATIVE, bool TO = false>
__global__ void __launch_bounds__(Epb<N, NC>::value * Shape<N>::NP)
    k_grad(long long E, const Ops* __restrict__ ops, PhysT<R> P, const R* __restrict__ geo,
           const R* __restrict__ fgeo, const int* __restrict__ nbr, const int* __restrict__ nbr_fo,
           const R* __restrict__ ug, const R* __restrict__ uf, R* __restrict__ qg, R* __restrict__ qf) {
  static_assert(!TO || NC == 1, "tangent-only gradient works on one plane");
  constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF, EPB = Epb<N, NC>::value, NT = EPB * NP, FT = EPB * 6 * NF;
  constexpr int NI = (FT + NT - 1) / NT;    // face points of a thread
  using V = Pack<NC, R>;
  __shared__ SmemOpsT<R> so;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* sU = reinterpret_cast<V*>(smem_raw);   // [5][NT]
  V* sUh = sU + 5 * NT;                     // [5][FT]
  V* sQ = sUh + 5 * FT;                     // [2][3][NT] gradient of the current variable and the last
  load_ops<N, R>(ops, so);
  const int tid = threadIdx.x, el = tid / NP, g = tid % NP;
  const long long e0 = (long long)blockIdx.x * EPB, e = e0 + el;
  const bool active = e < E;
  const long long plane_g = E * 5 * NP, plane_f = E * 30 * NF;
  const long long og = TO ? plane_g : 0, of = TO ? plane_f : 0;   // TO: the tangent plane
  // all loads are issued before the first is needed: neighbours, values (asynchronous copies), geometry of the
  // point's lines and of the face points at their ends (kept for all variables), traces
  int nb[NI], fo[NI];
#pragma unroll
  for (int it = 0; it < NI; ++it) {
    const int idx = tid + it * NT;
    const long long face = (e0 + idx / (6 * NF)) * 6 + (idx / NF) % 6;
    const bool ok = idx < FT && face < E * 6;
    nb[it] = ok ? nbr[face] : 0;
    fo[it] = ok ? nbr_fo[face] : 0;
  }
  if (active)
#pragma unroll
    for (int c = 0; c < 5; ++c)
#pragma unroll
      for (int p = 0; p < NC; ++p)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(sU + c * NT + tid) + p * (unsigned)sizeof(R)),
                     "l"(ug + og + p * plane_g + e * 5 * NP + c * NP + g), "n"(sizeof(R)) : "memory");
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  int lb[3], fp[3];
  R G[3][N][3], n[6][3], invW = R(0);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    lb[a] = g - ig[a] * pt_stride<N>(a);
    fp[a] = vol_face_point<N>(g, a);
  }
  if (active) {
    const R* gp = geo + e * 10 * NP;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int k = 0; k < N; ++k) G[a][k][d] = gp[(a * 3 + d) * NP + lb[a] + k * pt_stride<N>(a)];
#pragma unroll
        for (int side = 0; side < 2; ++side) n[2 * a + side][d] = fgeo[((e * 6 + 2 * a + side) * 4 + d) * NF + fp[a]];
      }
    invW = R(1) / gp[9 * NP + g];
  }
  // traces: u_hat on every face point (Eq. LDG2)
#pragma unroll
  for (int it = 0; it < NI; ++it) {
    const int idx = tid + it * NT;
    const int l = idx / (6 * NF), phi = (idx / NF) % 6, f = idx % NF;
    const long long ee = e0 + l;
    if (idx >= FT || ee >= E) continue;
    const long long fbase = ee * 30 * NF + phi * 5 * NF + f;
    const int f2 = orient_map((fo[it] >> 3) & 7, f % N, f / N, N);
    const long long nbase = nb[it] >= 0 ? (long long)nb[it] * 30 * NF + (fo[it] & 7) * 5 * NF + f2 : fbase;
    V own[5], oth[5];
#pragma unroll
    for (int c = 0; c < 5; ++c)
#pragma unroll
      for (int p = 0; p < NC; ++p) {
        own[c].v[p] = uf[of + p * plane_f + fbase + c * NF];
        oth[c].v[p] = uf[of + p * plane_f + nbase + c * NF];
      }
    V* dst = sUh + idx;
    if (nb[it] == -DG_BC_WALL) {
      const R sr = s_exp(R(0.5) * (TO ? uf[fbase] : own[0].v[0]));   // TO: the value plane's varrho trace
      V zero, last;
#pragma unroll
      for (int p = 0; p < NC; ++p) zero.v[p] = R(0);
      if constexpr (TO) {
        last.v[0] = R(0.5) * sr * P.t_wall * own[0].v[0];
      } else {
        last.v[0] = sr * P.t_wall;
        if constexpr (NC == 2) last.v[1] = R(0.5) * sr * P.t_wall * own[0].v[1];
      }
      dst[0] = own[0];
      dst[FT] = dst[2 * FT] = dst[3 * FT] = zero;
      dst[4 * FT] = last;
    } else {
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        V x;
#pragma unroll
        for (int p = 0; p < NC; ++p) x.v[p] = nb[it] >= 0 ? R(0.5) * (own[c].v[p] + oth[c].v[p]) : own[c].v[p];
        dst[c * FT] = x;
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  R D[3][N], ec[6];
  axis_coefs<N, true>(so.D, ig, D);
  end_coefs(so, ig, ec);
  R* qge = qg + (TO ? E * 15 * NP : 0) + e * 15 * NP + g;
#pragma unroll 1
  for (int c = 0; c < 5; ++c) {
    V* q = sQ + (c & 1) * 3 * NT;           // the other half is still being read for the traces
    if (active) {
      // q_d = (sum over the 6 faces of e_face[i_axis] (w n_d dS) u_hat_c - D^T (G u_c)) / (w |J|)
      V acc[3];
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int p = 0; p < NC; ++p) acc[d].v[p] = R(0);
#pragma unroll
      for (int phi = 0; phi < 6; ++phi) {
        const V uh = sUh[c * FT + (el * 6 + phi) * NF + fp[phi >> 1]];
#pragma unroll
        for (int d = 0; d < 3; ++d)
#pragma unroll
          for (int p = 0; p < NC; ++p) acc[d].v[p] = cm_fma<CM>(ec[phi], n[phi][d] * uh.v[p], acc[d].v[p]);
      }
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const V x = sU[c * NT + el * NP + lb[a] + k * pt_stride<N>(a)];
#pragma unroll
          for (int d = 0; d < 3; ++d)
#pragma unroll
            for (int p = 0; p < NC; ++p) acc[d].v[p] = cm_fma<CM>(-D[a][k], G[a][k][d] * x.v[p], acc[d].v[p]);
        }
#pragma unroll
      for (int d = 0; d < 3; ++d) {
#pragma unroll
        for (int p = 0; p < NC; ++p) {
          acc[d].v[p] = acc[d].v[p] * invW;
          qge[p * E * 15 * NP + (d * 5 + c) * NP] = acc[d].v[p];
        }
        q[d * NT + tid] = acc[d];
      }
    }
    __syncthreads();
    // both ends of a line per iteration
#pragma unroll
    for (int it = 0; it < (EPB * 3 * NF + NT - 1) / NT; ++it) {
      const int idx = tid + it * NT;
      const int l = idx / (3 * NF), a = (idx / NF) % 3, f = idx % NF;
      if (idx >= EPB * 3 * NF || e0 + l >= E) continue;
      const int base = l * NP + face_vol_point<N>(2 * a, f, 0);
      R* dst = qf + (TO ? E * 90 * NF : 0) + (e0 + l) * 90 * NF + a * 30 * NF + f;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        V end[2];
        line_ends<N, CM>(so, q + d * NT + base, pt_stride<N>(a), end);
#pragma unroll
        for (int side = 0; side < 2; ++side)
#pragma unroll
          for (int p = 0; p < NC; ++p) dst[p * E * 90 * NF + (side * 15 + d * 5 + c) * NF] = end[side].v[p];
      }
    }
  }
}

// --------------------------------------------------------------------------------------------
// k_faces: numerical flux of Eq. LDG2 on every face, written for both element faces
// --------------------------------------------------------------------------------------------
template <typename S, int NC, typename R>
__device__ __forceinline__ S ld(const R* p, long long plane) {
  if constexpr (NC == 1) return p[0];
  else return S{p[0], p[plane]};
}
template <typename R>
__device__ __forceinline__ void st(R* p, long long, R v) { p[0] = v; }
template <typename R>
__device__ __forceinline__ void st(R* p, long long plane, DualT<R> v) {
  p[0] = v.v;
  p[plane] = v.d;
}

// interior numerical flux of Eq. LDG2 with the normal n = w n dS of the first side:
// F_hat . n = (F(u, q) + F(u2, q2)) . n / 2 + sigma(u_hat) (u - u_hat) |n|, u_hat = (u + u2) / 2
template <typename S, typename R = typename RealOf<S>::type>
__device__ __forceinline__ void face_flux_interior(const PhysT<R>& P, const S u[5], const S q[3][5], const S u2[5],
                                                   const S q2[3][5], const R n[3], R area, S out[5],
                                                   const Mix<R>& mx) {
  S f1[5], fn[5], uh[5], sg[5];
  flux_dot_n(P, u, q, n, true, f1, mx);
  flux_dot_n(P, u2, q2, n, true, fn, mx);
#pragma unroll
  for (int c = 0; c < 5; ++c) uh[c] = R(0.5) * (u[c] + u2[c]);
  sigma_diag(P, uh, sg, mx);
#pragma unroll
  for (int c = 0; c < 5; ++c) out[c] = R(0.5) * (f1[c] + fn[c]) + sg[c] * ((R(0.5) * area) * (u[c] - u2[c]));
}

// vout false (NC = 2): only the flux's tangent is written, r being unwanted
template <int N, int NC, typename R>
__global__ void k_faces(long long E, long long F, PhysT<R> P, const int* __restrict__ face_e,
                        const int* __restrict__ face_f, const int* __restrict__ nbr,
                        const int* __restrict__ nbr_fo, const R* __restrict__ fgeo,
                        const R* __restrict__ uf, const R* __restrict__ qf,
                        R* __restrict__ fh, const R* __restrict__ mixf, bool vout) {
  auto put = [&](R* p, long long plane, const auto& x) {
    if constexpr (NC == 1) {
      p[0] = x;
    } else {
      if (vout) p[0] = x.v;
      p[plane] = x.d;
    }
  };
  using S = typename std::conditional<NC == 2, DualT<R>, R>::type;
  constexpr int NF = Shape<N>::NF;
  const long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= F * NF) return;
  const long long fi = idx / NF;
  const int f = (int)(idx % NF);
  const long long e = face_e[fi];
  const int phi = face_f[fi];
  Mix<R> mx{P.cv, R(1)};
  if (P.comp) {   // mixture at this face point: [E][6][2][NF] = (c_v*, conductivity factor)
    mx.cv = mixf[((e * 6 + phi) * 2) * NF + f];
    mx.kfac = mixf[((e * 6 + phi) * 2 + 1) * NF + f];
  }
  const long long plane_u = E * 30 * NF, plane_q = E * 90 * NF;
  const R* gp = fgeo + ((e * 6 + phi) * 4) * NF + f;
  const R n[3] = {gp[0], gp[NF], gp[2 * NF]};
  const R area = gp[3 * NF];
  S u[5], q[3][5];
  const long long ub = e * 30 * NF + phi * 5 * NF + f;
  const long long qb = e * 90 * NF + phi * 15 * NF + f;
#pragma unroll
  for (int c = 0; c < 5; ++c) u[c] = ld<S, NC, R>(uf + ub + c * NF, plane_u);
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int c = 0; c < 5; ++c) q[d][c] = ld<S, NC, R>(qf + qb + (d * 5 + c) * NF, plane_q);
  const int nb = nbr[e * 6 + phi];
  S out[5];
  if (nb >= 0) {
    const int fo = nbr_fo[e * 6 + phi];
    const int phi2 = fo & 7;
    const int f2 = orient_map(fo >> 3, f % N, f / N, N);
    S u2[5], q2[3][5];
    const long long ub2 = (long long)nb * 30 * NF + phi2 * 5 * NF + f2;
    const long long qb2 = (long long)nb * 90 * NF + phi2 * 15 * NF + f2;
#pragma unroll
    for (int c = 0; c < 5; ++c) u2[c] = ld<S, NC, R>(uf + ub2 + c * NF, plane_u);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int c = 0; c < 5; ++c) q2[d][c] = ld<S, NC, R>(qf + qb2 + (d * 5 + c) * NF, plane_q);
    const long long ob2 = (long long)nb * 30 * NF + phi2 * 5 * NF + f2;
    face_flux_interior(P, u, q, u2, q2, n, area, out, mx);
#pragma unroll
    for (int c = 0; c < 5; ++c) put(fh + ob2 + c * NF, plane_u, -out[c]);
  } else if (nb == -DG_BC_WALL) {
    S ubd[5], sg[5];
    wall_trace(P, u, ubd);
    flux_dot_n(P, ubd, q, n, true, out, mx);
    sigma_diag(P, ubd, sg, mx);
#pragma unroll
    for (int c = 0; c < 5; ++c) out[c] = out[c] + sg[c] * (area * (u[c] - ubd[c]));
  } else {
    flux_dot_n(P, u, q, n, false, out, mx);
  }
#pragma unroll
  for (int c = 0; c < 5; ++c) put(fh + ub + c * NF, plane_u, out[c]);
}

// --------------------------------------------------------------------------------------------
// k_volume: pointwise flux and source, projection, lifting of F_hat, B^T -> nodal r (and J v)
// --------------------------------------------------------------------------------------------
template <typename S, typename R = typename RealOf<S>::type>
__device__ __forceinline__ void volume_point(const PhysT<R>& P, const S u[5], const S q[3][5],
                                             const R G[9], R Wd, const R acc[3],
                                             const R* xg, R t, S Fref[3][5], S src[5], const R mg[8]) {
  // mg (variable composition): c_v*, grad c_v* (3), conductivity factor, mass fractions of N2, O2, He
  const Mix<R> mx{P.comp ? mg[0] : P.cv, P.comp ? mg[4] : R(1)};
  const R cvp = mx.cv;
  const R pcoef = P.comp ? cvp * P.inv_gamma : P.p_coef;   // 1/(gamma m*)
  Prim<S> w;
  primitives(P, u, q, w, mx);
  const S cm = (P.c_mu * w.mu) * w.isr;
  const S ck = ((P.c_k / cvp) * w.kappa) * w.isr;
  // reference-space fluxes Fref[a][c] = sum_d G[a][d] F[c][d], formed from the contractions of the
  // cofactor rows with v, grad T and the strain rows (F[c][d] = u_c v_d + p delta - viscous terms)
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const R g0 = G[a * 3 + 0], g1 = G[a * 3 + 1], g2 = G[a * 3 + 2];
    const S Gv = g0 * w.v[0] + g1 * w.v[1] + g2 * w.v[2];
    const S GgT = g0 * w.gT[0] + g1 * w.gT[1] + g2 * w.gT[2];
    Fref[a][0] = u[0] * Gv;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const S Ge = g0 * w.eps[m][0] + g1 * w.eps[m][1] + g2 * w.eps[m][2];
      Fref[a][1 + m] = u[1 + m] * Gv + (pcoef * G[a * 3 + m]) * u[4] - cm * Ge;
    }
    Fref[a][4] = u[4] * Gv - ck * GgT;
  }
  // source terms
  const S sr = s_inv(w.isr);
  const S wxv[3] = {P.omega[1] * w.v[2] - P.omega[2] * w.v[1], P.omega[2] * w.v[0] - P.omega[0] * w.v[2],
                    P.omega[0] * w.v[1] - P.omega[1] * w.v[0]};
  src[0] = (u[0] - R(1)) * w.div;
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    const S a_m = acc[m] - P.cor * wxv[m];
    const S eg = w.eps[m][0] * q[0][0] + w.eps[m][1] * q[1][0] + w.eps[m][2] * q[2][0];
    src[1 + m] = sr * a_m + R(0.5) * (w.div * u[1 + m]) - (R(0.5) * pcoef) * (u[4] * q[m][0]) + R(0.5) * (cm * eg);
  }
  const S tg = w.gT[0] * q[0][0] + w.gT[1] * q[1][0] + w.gT[2] * q[2][0];
  S diss = s_zero<S>();
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int d = 0; d < 3; ++d) diss = diss + w.eps[m][d] * w.gv[m][d];
  S s4 = (R(1.5) - P.gamma) * (u[4] * w.div) + R(0.5) * (ck * tg) + ((P.c_d / cvp) * w.mu) * (w.isr * diss);
  if (P.comp) {
    // -(1/c_v) (sqrt(rho) T v - c_kappa kappa / (sqrt(rho) c_v) grad T) . grad c_v
    const S vg = w.v[0] * mg[1] + w.v[1] * mg[2] + w.v[2] * mg[3];
    const S tgc = w.gT[0] * mg[1] + w.gT[1] * mg[2] + w.gT[2] * mg[3];
    s4 = s4 - (u[4] * vg - ck * tgc) * (R(1) / cvp);
  }
  if (P.euv == DG_EUV_GAUSS) {
    const R r = sqrt(xg[0] * xg[0] + xg[1] * xg[1] + xg[2] * xg[2]);
    const R sx = cos(P.euv_omega_t * t), sy = -sin(P.euv_omega_t * t);
    R cchi = (xg[0] * sx + xg[1] * sy) / r;
    cchi = fmin(R(1), fmax(R(-1), cchi));
    const R chi = acos(cchi);
    const R dz = (r - P.euv_r_peak) * P.euv_inv_w;
    const R Qh = P.euv_amp * s_exp(-chi * chi * P.euv_inv2s2) * s_exp(R(-0.6931471805599453) * dz * dz);
    s4 = s4 + (Qh / cvp) * w.isr;
  } else if (P.euv == DG_EUV_EUVAC) {
    // EUVAC photoabsorption with Smith & Smith Chapman depths (Sec. 2.2)
    const R r = sqrt(xg[0] * xg[0] + xg[1] * xg[1] + xg[2] * xg[2]);
    const R wt = P.euv_omega_t * t;
    R cchi = (xg[0] * (-P.sun_cd * cos(wt)) + xg[1] * (P.sun_cd * sin(wt)) + xg[2] * P.sun_sd) / r;
    cchi = fmin(R(1), fmax(R(-1), cchi));
    const R schi = sqrt(fmax(R(0), R(1) - cchi * cchi));
    if (cchi > R(0) || schi * r > P.g_r0) {          // not in the Earth's shadow
      const S er = sr * sr;                             // e^varrho
      const R minv = P.comp ? cvp : P.inv_m;            // 1/m*
      const S Hs = w.T * (r * r * minv / (P.g_r0 * P.g_r0));   // H* = T* r*^2 / (m* g_r0^2)
      const S rt = r * s_inv(Hs);                       // r~ = |r| / H
      const S ex = s_erfcx(s_sqrt(R(0.5) * rt) * fabs(cchi));
      const S base = s_sqrt(R(1.5707963267948966) * rt);
      S ch;
      if (cchi > R(0)) ch = base * ex;
      else ch = base * (R(2) * s_exp(rt * (R(1) - schi)) - ex);
      // species weights w_s = chi_s / m_s* (O, N2, O2, He), or 1/m* on oxygen alone
      R ws[4] = {P.inv_m, R(0), R(0), R(0)};
      if (P.comp) {
        ws[0] = (R(1) - mg[5] - mg[6] - mg[7]);
        ws[1] = mg[5] * R(16.0 / 28.0);
        ws[2] = mg[6] * R(16.0 / 32.0);
        ws[3] = mg[7] * R(16.0 / 4.0);
      }
      const S k = (P.euvac_cc * er) * Hs * ch;          // tau_j = Phi_j k
      S qs = s_zero<S>();
#pragma unroll 1
      for (int j = 0; j < P.n_euvac; ++j) {
        const R Phi = ws[0] * P.euvac_phi[0][j] + ws[1] * P.euvac_phi[1][j] + ws[2] * P.euvac_phi[2][j] +
                      ws[3] * P.euvac_phi[3][j];
        qs = qs + (P.euvac_B[j] * Phi) * s_exp(-Phi * k);
      }
      s4 = s4 + (er * qs) * (R(1) / cvp) * w.isr;
    }
  }
  src[4] = s4;
#pragma unroll
  for (int c = 0; c < 5; ++c) src[c] = src[c] * Wd;
}

// L2 prefetch hint for n consecutive elements from p, one 128-byte line per thread and iteration
template <typename R>
__device__ __forceinline__ void prefetch_l2(const R* p, long long n) {
  const char* c = reinterpret_cast<const char*>(p);
  const long long bytes = n * (long long)sizeof(R);
  for (long long off = threadIdx.x * 128LL; off < bytes; off += blockDim.x * 128LL)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(c + off));
}

// stage_c != 0 (NC = 2): the tangent output is the DIRK stage operator J_G v = M v - stage_c J_r v,
// M v = B^T (W B v) being formed from the tangent's own Gauss values
// FP32: at least two CTAs per SM (four for the p = 3 Jv, where 128 registers suffice without spills), since
// the value + tangent physics would otherwise take enough registers to halve the resident warps of
// this latency-bound kernel (FP64 is bound by its pipe instead)
template <int OUT, typename R>
__device__ __forceinline__ Pack<OUT, R> planes_of(R x) { return {x}; }
template <int OUT, typename R>
__device__ __forceinline__ Pack<OUT, R> planes_of(DualT<R> x) {
  Pack<OUT, R> y;
  if constexpr (OUT == 2) y.v[0] = x.v;
  y.v[OUT - 1] = x.d;
  return y;
}

// OUT planes leave the kernel: NC, or 1 of the 2 (r not wanted: the tangent alone is contracted)
template <int N, int NC, int OUT, typename R, int CM = CM_NATIVE>
__global__ void __launch_bounds__(Epb<N, NC>::value * Shape<N>::NP, N == 4 && NC == 2 ? 4 : 2)
k_volume(long long E, const Ops* __restrict__ ops, PhysT<R> P, R t,
                         const R* __restrict__ geo, const R* __restrict__ accg,
                         const R* __restrict__ xg, const R* __restrict__ ug,
                         const R* __restrict__ qg, const R* __restrict__ fh,
                         double* __restrict__ r, double* __restrict__ jv, R stage_c,
                         const R* __restrict__ mixg, long long ahead) {
  using S = typename std::conditional<NC == 2, DualT<R>, R>::type;
  constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF, EPB = Epb<N, NC>::value;
  constexpr int NT = EPB * NP, FT = EPB * 6 * NF;
  using V = Pack<OUT, R>;
  __shared__ SmemOpsT<R> so;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  V* sF = reinterpret_cast<V*>(smem_raw);   // [15][NT]  reference fluxes a * 5 + c
  V* sH = sF + 15 * NT;                     // [5][FT]   face fluxes
  V* sR = sH + 5 * FT;                      // [5][NT]
  load_ops<N, R>(ops, so);
  const long long e0 = (long long)blockIdx.x * EPB;
  if constexpr (sizeof(R) == 4) {
    // FP32 is latency-bound on these loads: pull into L2 the records of the CTA `ahead` launches
    // later (one residency wave, so it starts about when this one ends)
    const long long eb = e0 + ahead * EPB;
    if (ahead > 0 && eb < E) {
      const long long ne = (E - eb < EPB) ? E - eb : EPB;
      for (int pl = 0; pl < NC; ++pl) {
        prefetch_l2(ug + pl * E * 5 * NP + eb * 5 * NP, ne * 5 * NP);
        prefetch_l2(qg + pl * E * 15 * NP + eb * 15 * NP, ne * 15 * NP);
        if (pl >= NC - OUT) prefetch_l2(fh + pl * E * 30 * NF + eb * 30 * NF, ne * 30 * NF);
      }
      prefetch_l2(geo + eb * 10 * NP, ne * 10 * NP);
      prefetch_l2(accg + eb * 3 * NP, ne * 3 * NP);
      if (P.euv) prefetch_l2(xg + eb * 3 * NP, ne * 3 * NP);
      if (P.comp) prefetch_l2(mixg + eb * 8 * NP, ne * 8 * NP);
    }
  }
  const long long plane_f = E * 30 * NF;
  for (int idx = threadIdx.x; idx < EPB * 30 * NF; idx += NT) {
    const int l = idx / (30 * NF), rem = idx % (30 * NF);
    const long long ee = e0 + l;
    if (ee < E) {
      const int phi = rem / (5 * NF), c = (rem / NF) % 5, f = rem % NF;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(sH + c * FT + (l * 6 + phi) * NF + f);
#pragma unroll
      for (int p = 0; p < OUT; ++p)         // arrives while the pointwise physics runs (232 -> 188 us)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst + p * (unsigned)sizeof(R)),
                     "l"(fh + (NC - OUT + p) * plane_f + ee * 30 * NF + rem), "n"(sizeof(R)) : "memory");
    }
  }
  const int tid = threadIdx.x, el = tid / NP, g = tid % NP;
  const long long e = e0 + el;
  const bool active = e < E;
  S srcv[5];
  R wu[5] = {R(0), R(0), R(0), R(0), R(0)};   // W u_dot at this point (stage operator)
  if (active) {
    const long long plane_g = E * 5 * NP, plane_q = E * 15 * NP;
    S u[5], q[3][5];
#pragma unroll
    for (int c = 0; c < 5; ++c) u[c] = ld<S, NC, R>(ug + e * 5 * NP + c * NP + g, plane_g);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int c = 0; c < 5; ++c) q[d][c] = ld<S, NC, R>(qg + e * 15 * NP + (d * 5 + c) * NP + g, plane_q);
    R G[9];
    const R* gp = geo + e * 10 * NP + g;
#pragma unroll
    for (int k = 0; k < 9; ++k) G[k] = gp[k * NP];
    const R Wd = gp[9 * NP];
    const R a3[3] = {accg[e * 3 * NP + g], accg[e * 3 * NP + NP + g], accg[e * 3 * NP + 2 * NP + g]};
    R x3[3] = {R(0), R(0), R(0)};
    if (P.euv) {
      x3[0] = xg[e * 3 * NP + g];
      x3[1] = xg[e * 3 * NP + NP + g];
      x3[2] = xg[e * 3 * NP + 2 * NP + g];
    }
    S Fref[3][5];
    R mg[8] = {R(0), R(0), R(0), R(0), R(0), R(0), R(0), R(0)};
    if (P.comp) {
#pragma unroll
      for (int k = 0; k < 8; ++k) mg[k] = mixg[(e * 8 + k) * NP + g];
    }
    volume_point<S>(P, u, q, G, Wd, a3, x3, t, Fref, srcv, mg);
    if constexpr (NC == 2) {
#pragma unroll
      for (int c = 0; c < 5; ++c) wu[c] = Wd * u[c].d;
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int c = 0; c < 5; ++c) sF[(a * 5 + c) * NT + tid] = planes_of<OUT>(Fref[a][c]);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const int ig[3] = {g % N, (g / N) % N, g / (N * N)};
  if (active) {
    R D[3][N], ec[6];
    axis_coefs<N, true>(so.D, ig, D);
    end_coefs(so, ig, ec);
    int fp[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) fp[a] = el * 6 * NF + vol_face_point<N>(g, a);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      V acc = planes_of<OUT>(srcv[c]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int st = pt_stride<N>(a);
        const V* y = sF + (a * 5 + c) * NT + tid - ig[a] * st;
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const V x = y[k * st];
#pragma unroll
          for (int p = 0; p < OUT; ++p) acc.v[p] = cm_fma<CM>(D[a][k], x.v[p], acc.v[p]);
        }
      }
#pragma unroll
      for (int phi = 0; phi < 6; ++phi) {
        const V x = sH[c * FT + phi * NF + fp[phi >> 1]];
#pragma unroll
        for (int p = 0; p < OUT; ++p) acc.v[p] = cm_fma<CM>(-ec[phi], x.v[p], acc.v[p]);
      }
      if (NC == 2 && stage_c != R(0)) acc.v[OUT - 1] = wu[c] - stage_c * acc.v[OUT - 1];
      sR[c * NT + tid] = acc;
    }
  }
  __syncthreads();
  V *in = sR, *out = sF;                    // the fluxes have been read
#pragma unroll
  for (int dir = 0; dir < 3; ++dir) {
    const int st = pt_stride<N>(dir), base = tid - ig[dir] * st;
    R B[N];
#pragma unroll
    for (int k = 0; k < N; ++k) B[k] = so.B[k * N + ig[dir]];
    if (active)
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        V acc;
#pragma unroll
        for (int p = 0; p < OUT; ++p) acc.v[p] = R(0);
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const V x = in[c * NT + base + k * st];
#pragma unroll
          for (int p = 0; p < OUT; ++p) acc.v[p] = cm_fma<CM>(B[k], x.v[p], acc.v[p]);
        }
        if (dir < 2) {
          out[c * NT + tid] = acc;
        } else {
          const long long o = e * 5 * NP + c * NP + g;
          if (OUT == NC && r) r[o] = as_f64(acc.v[0]);
          if (NC == 2) jv[o] = as_f64(acc.v[OUT - 1]);
        }
      }
    if (dir < 2) __syncthreads();
    V* tt = in;
    in = out;
    out = tt;
  }
}

}  // namespace dg

#include "dg_fp64.cuh"
#include "dg_blocks.cuh"

namespace dg {

// variable composition (Sec. 2.1.1-2.1.2) at the Gauss and face points from the positions xg:
// mixg [E][8][NP] = (c_v*, grad c_v* (3), conductivity factor, chi_N2, chi_O2, chi_He),
// mixf [E][6][2][NF] = (c_v*, conductivity factor); face positions are the exact extrapolation of
// the Gauss-point positions (the map is a polynomial of degree p)
__device__ inline void mixture_at(const Phys& P, const double x[3], double out[8]) {
  const double r = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
  const double inv_ms[4] = {1.0, 16.0 / 28.0, 16.0 / 32.0, 16.0 / 4.0};      // m_O / m_s
  const double alpha[4] = {1.0, 3.6 / 5.6, 3.6 / 5.6, 1.0};                  // alpha_s / alpha_O
  double chi[4], dchi[4];
  chi[0] = 1.0;
  dchi[0] = 0.0;
  for (int s = 0; s < 3; ++s) {
    double c = 0.0, dc = 0.0;
    for (int j = 0; j < 2; ++j) {
      const double t = P.comp_a[2 * s + j] * exp(P.comp_b[2 * s + j] * r);
      c += t;
      dc += P.comp_b[2 * s + j] * t;
    }
    chi[1 + s] = c;
    dchi[1 + s] = dc;
    chi[0] -= c;
    dchi[0] -= dc;
  }
  double cv = 0.0, dcv = 0.0, ka = 0.0;
  for (int s = 0; s < 4; ++s) {
    cv += chi[s] * inv_ms[s];
    dcv += dchi[s] * inv_ms[s];
    ka += chi[s] * inv_ms[s] * alpha[s];
  }
  out[0] = cv;
  for (int d = 0; d < 3; ++d) out[1 + d] = dcv * x[d] / r;
  out[4] = ka / cv;
  out[5] = chi[1];
  out[6] = chi[2];
  out[7] = chi[3];
}

template <int N>
__global__ void k_mixture(long long E, const Ops* __restrict__ ops, Phys P, const double* __restrict__ xg,
                          double* __restrict__ mixg, double* __restrict__ mixf) {
  constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF;
  const long long e = blockIdx.x;
  if (e >= E) return;
  for (int g = threadIdx.x; g < NP; g += blockDim.x) {
    const double x[3] = {xg[(e * 3 + 0) * NP + g], xg[(e * 3 + 1) * NP + g], xg[(e * 3 + 2) * NP + g]};
    double o[8];
    mixture_at(P, x, o);
    for (int k = 0; k < 8; ++k) mixg[(e * 8 + k) * NP + g] = o[k];
  }
  for (int idx = threadIdx.x; idx < 6 * NF; idx += blockDim.x) {
    const int phi = idx / NF, f = idx % NF;
    const double* ev = (phi & 1) ? ops->eR : ops->eL;
    double x[3] = {0.0, 0.0, 0.0};
    for (int d = 0; d < 3; ++d)
      for (int k = 0; k < N; ++k) x[d] = fma(ev[k], xg[(e * 3 + d) * NP + face_vol_point<N>(phi, f, k)], x[d]);
    double o[8];
    mixture_at(P, x, o);
    mixf[((e * 6 + phi) * 2) * NF + f] = o[0];
    mixf[((e * 6 + phi) * 2 + 1) * NF + f] = o[4];
  }
}

// --------------------------------------------------------------------------------------------
// geometry at Gauss points and face points (isoparametric map of the node coordinates)
// --------------------------------------------------------------------------------------------
// UNW: gu and fgu, without weights, for the FP64 kernels; else geo, acc, xg and fgeo
template <int N, bool UNW>
__global__ void k_geometry(long long E, const Ops* __restrict__ ops, Phys P, int gravity_kind,
                           double g0, double g1, double g2, double g_r0,
                           const double* __restrict__ x, double* __restrict__ geo,
                           double* __restrict__ accg, double* __restrict__ xg, double* __restrict__ fgeo,
                           double* __restrict__ gu, double* __restrict__ fgu) {
  constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF;
  __shared__ SmemOps so;
  __shared__ double w1[MAXN];
  extern __shared__ double smem[];
  double* b0 = smem;           // [3][NP]
  double* b1 = b0 + 3 * NP;    // [3][NP]
  double* J = b1 + 3 * NP;     // [9][NP] J[d][a]
  load_ops<N, double>(ops, so);
  if (threadIdx.x < N) w1[threadIdx.x] = ops->w[threadIdx.x];
  const long long e = blockIdx.x;
  const int g = threadIdx.x;
  // positions relative to the element's first node: the Jacobian is unchanged (derivatives of the
  // basis sum to zero) and its rounding is relative to the element size instead of |x|
  for (int idx = threadIdx.x; idx < 3 * NP; idx += blockDim.x) {
    const int c = idx / NP;
    b0[idx] = x[e * 3 * NP + idx] - x[e * 3 * NP + c * NP];
  }
  __syncthreads();
  double* in = b0;
  double* out = b1;
  for (int dir = 0; dir < 3; ++dir) {
    if (g < NP)
      for (int c = 0; c < 3; ++c) out[c * NP + g] = line<N, false>(so.B, in + c * NP, g, dir);
    __syncthreads();
    double* tt = in;
    in = out;
    out = tt;
  }
  // in: Gauss point positions relative to the first node
  if (g < NP) {
    for (int d = 0; d < 3; ++d)
      for (int a = 0; a < 3; ++a) J[(d * 3 + a) * NP + g] = line<N, false>(so.D, in + d * NP, g, a);
  }
  __syncthreads();
  if (g < NP) {
    double j[3][3];
    for (int d = 0; d < 3; ++d)
      for (int a = 0; a < 3; ++a) j[d][a] = J[(d * 3 + a) * NP + g];
    // cofactors: cof[d][a] = d(det)/d j[d][a] = det * (J^{-1})[a][d]
    double cof[3][3];
    cof[0][0] = j[1][1] * j[2][2] - j[1][2] * j[2][1];
    cof[0][1] = j[1][2] * j[2][0] - j[1][0] * j[2][2];
    cof[0][2] = j[1][0] * j[2][1] - j[1][1] * j[2][0];
    cof[1][0] = j[0][2] * j[2][1] - j[0][1] * j[2][2];
    cof[1][1] = j[0][0] * j[2][2] - j[0][2] * j[2][0];
    cof[1][2] = j[0][1] * j[2][0] - j[0][0] * j[2][1];
    cof[2][0] = j[0][1] * j[1][2] - j[0][2] * j[1][1];
    cof[2][1] = j[0][2] * j[1][0] - j[0][0] * j[1][2];
    cof[2][2] = j[0][0] * j[1][1] - j[0][1] * j[1][0];
    const double det = j[0][0] * cof[0][0] + j[0][1] * cof[0][1] + j[0][2] * cof[0][2];
    const int i0 = g % N, i1 = (g / N) % N, i2 = g / (N * N);
    const double wq = w1[i0] * w1[i1] * w1[i2];
    if constexpr (UNW) {
      double* gq = gu + e * 11 * NP + g;
      for (int a = 0; a < 3; ++a)
        for (int d = 0; d < 3; ++d) gq[(a * 3 + d) * NP] = cof[d][a];
      gq[9 * NP] = det;
      gq[10 * NP] = 1.0 / det;
    } else {
      double* gp = geo + e * 10 * NP + g;
      for (int a = 0; a < 3; ++a)
        for (int d = 0; d < 3; ++d) gp[(a * 3 + d) * NP] = wq * cof[d][a];
      gp[9 * NP] = wq * det;
      const double X[3] = {x[e * 3 * NP] + in[g], x[e * 3 * NP + NP] + in[NP + g], x[e * 3 * NP + 2 * NP] + in[2 * NP + g]};
      for (int d = 0; d < 3; ++d) xg[e * 3 * NP + d * NP + g] = X[d];
      double gv[3];
      if (gravity_kind == 0) {
        gv[0] = g0; gv[1] = g1; gv[2] = g2;
      } else {
        const double rr = sqrt(X[0] * X[0] + X[1] * X[1] + X[2] * X[2]);
        const double fac = -(g_r0 / rr) * (g_r0 / rr) / rr;
        for (int d = 0; d < 3; ++d) gv[d] = fac * X[d];
      }
      const double* w = P.omega;
      const double wx[3] = {w[1] * X[2] - w[2] * X[1], w[2] * X[0] - w[0] * X[2], w[0] * X[1] - w[1] * X[0]};
      const double wwx[3] = {w[1] * wx[2] - w[2] * wx[1], w[2] * wx[0] - w[0] * wx[2], w[0] * wx[1] - w[1] * wx[0]};
      const double cen = (P.cor * P.cor * 0.25);   // Fr^2 (cor = 2 Fr / sqrt(gamma))
      for (int d = 0; d < 3; ++d) accg[e * 3 * NP + d * NP + g] = gv[d] / P.gamma - cen * wwx[d];
    }
  }
  // faces: extrapolate the tangential Jacobian columns, n dS = side * (J_{a+1} x J_{a+2})
  for (int idx = threadIdx.x; idx < 6 * NF; idx += blockDim.x) {
    const int phi = idx / NF, f = idx % NF;
    const int axis = phi >> 1;
    const double side = (phi & 1) ? 1.0 : -1.0;
    const double* ev = (phi & 1) ? so.eR : so.eL;
    const int a1 = (axis + 1) % 3, a2 = (axis + 2) % 3;
    double t1[3], t2[3];
    for (int d = 0; d < 3; ++d) {
      double s1 = 0.0, s2 = 0.0;
      for (int k = 0; k < N; ++k) {
        const int gg = face_vol_point<N>(phi, f, k);
        s1 = fma(ev[k], J[(d * 3 + a1) * NP + gg], s1);
        s2 = fma(ev[k], J[(d * 3 + a2) * NP + gg], s2);
      }
      t1[d] = s1;
      t2[d] = s2;
    }
    double nv[3] = {t1[1] * t2[2] - t1[2] * t2[1], t1[2] * t2[0] - t1[0] * t2[2], t1[0] * t2[1] - t1[1] * t2[0]};
    const int is = f % N, it = f / N;
    const double wf = w1[is] * w1[it];
    double a2n = 0.0;
    if constexpr (UNW) {
      double* fq = fgu + ((e * 6 + phi) * 4) * NF + f;
      for (int d = 0; d < 3; ++d) {
        fq[d * NF] = side * nv[d];
        a2n += nv[d] * nv[d];
      }
      fq[3 * NF] = sqrt(a2n);
    } else {
      double* fp = fgeo + ((e * 6 + phi) * 4) * NF + f;
      for (int d = 0; d < 3; ++d) {
        fp[d * NF] = wf * side * nv[d];
        a2n += nv[d] * nv[d];
      }
      fp[3 * NF] = wf * sqrt(a2n);
    }
  }
}

// --------------------------------------------------------------------------------------------
// Driver
// --------------------------------------------------------------------------------------------
template <int N, int NC, typename R>
struct Smem {
  static constexpr int NP = Shape<N>::NP, NF = Shape<N>::NF, C = 5 * NC, EPB = Epb<N, NC>::value;
  static constexpr size_t interp = sizeof(R) * (2 * EPB * C * NP);
  static constexpr size_t grad = sizeof(R) * NC * EPB * (11 * NP + 30 * NF);
  static constexpr size_t volume = sizeof(R) * EPB * (20 * NP + 30 * NF);   // per output plane
};

template <typename R> inline WorkT<R> work_of(dg_mesh* m);
template <> inline WorkT<double> work_of<double>(dg_mesh* m) {
  return WorkT<double>{m->ws.ug, m->ws.uf, m->ws.qg, m->ws.qf, m->ws.fh, m->geo, m->fgeo, m->acc, m->xg,
                       m->mixg, m->mixf};
}
template <> inline WorkT<float> work_of<float>(dg_mesh* m) { return m->w32; }

// The limit is a property of the kernel in the whole process, so every caller sets the same value, the size of the
// instance's largest launch: with each call's own size, a thread working on a small mesh could lower it between
// another thread's call and its launch, which was then refused.
template <typename K>
static int set_smem(K kernel, size_t bytes) {
  cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (err != cudaSuccess) return fail(DG_ECUDA, std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(err));
  return DG_OK;
}

// FP64: `planes` planes from plane `first` on (u -> first, v -> the next) with k_interp64
template <int N>
static int launch_interp64(dg_mesh* m, const double* u, const double* v, int first, cudaStream_t s) {
  using G = Grp<N>;
  const int threads = threads64<N>(m->E * (v ? 2 : 1)), per = threads / G::T;
  const size_t sm = sizeof(cell) * 10 * G::NP * per;
  int rc = set_smem(k_interp64<N, false>, sizeof(cell) * 10 * G::NP * groups64_max<N>());
  if (rc) return rc;
  prof_begin(m, s, KK_INTERP);
  k_interp64<N, false><<<dim3((unsigned)((m->E + per - 1) / per), v ? 2 : 1), threads, sm, s>>>(
      u, v, m->E, m->d_ops, m->ws.ug + first * m->E * 5 * G::NP, m->ws.uf + first * m->E * 30 * G::NF);
  prof_end(m, s);
  DG_LAUNCH_CHECK("k_interp64");
  return DG_OK;
}

template <int N, int NC, typename R = double, int CM = CM_NATIVE>
static int run_interp(dg_mesh* m, const double* u, const double* v, cudaStream_t s) {
  constexpr int EPB = Epb<N, NC>::value, NP = Shape<N>::NP;
  if constexpr (std::is_same<R, double>::value) {
    if (m->interp_mode == DG_INTERP_TC) return interp_tc<N, NC>(m, u, v, m->ws.ug, m->ws.uf, s);
    return launch_interp64<N>(m, u, NC == 2 ? v : nullptr, 0, s);
  } else {
    const size_t sm = Smem<N, NC, R>::interp;
    int rc = set_smem(k_interp<N, NC, R, CM>, sm);
    if (rc) return rc;
    const unsigned blocks = (unsigned)((m->E + EPB - 1) / EPB);
    const WorkT<R> w = work_of<R>(m);
    prof_begin(m, s, KK_INTERP);
    k_interp<N, NC, R, CM><<<blocks, EPB * NP, sm, s>>>(u, v, m->E, m->d_ops, w.ug, w.uf);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_interp");
    return DG_OK;
  }
}

template <int N, int NC, typename R = double, int CM = CM_NATIVE, bool TO = false>
static int run_grad(dg_mesh* m, cudaStream_t s) {
  if constexpr (std::is_same<R, double>::value) {
    using G = Grp<N>;
    const int threads = threads64<N>(m->E * NC), per = threads / G::T;
    const size_t sm = sizeof(cell) * GradCells<N>::size * per;
    int rc = set_smem(k_grad64<N>, sizeof(cell) * GradCells<N>::size * groups64_max<N>());
    if (rc) return rc;
    prof_begin(m, s, KK_GRAD);
    k_grad64<N><<<dim3((unsigned)((m->E + per - 1) / per), NC), threads, sm, s>>>(
        m->E, m->d_ops, m->phys.t_wall, TO ? 1 : 0, m->gu, m->fgu, m->nbr, m->nbr_fo, m->ws.ug, m->ws.uf,
        m->ws.qg, m->ws.qf);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_grad64");
    return DG_OK;
  } else {
    constexpr int EPB = Epb<N, NC>::value, NP = Shape<N>::NP;
    const size_t sm = Smem<N, NC, R>::grad;
    int rc = set_smem(k_grad<N, NC, R, CM, TO>, sm);
    if (rc) return rc;
    const unsigned blocks = (unsigned)((m->E + EPB - 1) / EPB);
    const WorkT<R> w = work_of<R>(m);
    prof_begin(m, s, KK_GRAD);
    k_grad<N, NC, R, CM, TO><<<blocks, EPB * NP, sm, s>>>(m->E, m->d_ops, phys_as<R>(m->phys), w.geo, w.fgeo,
                                                            m->nbr, m->nbr_fo, w.ug, w.uf, w.qg, w.qf);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_grad");
    return DG_OK;
  }
}

// the tangent plane of ug, uf (nodal v -> Gauss values and traces), with the NC = 1 kernel
template <int N, typename R>
static int run_interp_tangent(dg_mesh* m, const double* v, cudaStream_t s) {
  constexpr int EPB = Epb<N, 1>::value, NP = Shape<N>::NP, NF = Shape<N>::NF;
  if constexpr (std::is_same<R, double>::value) {
    if (m->interp_mode == DG_INTERP_TC)
      return interp_tc<N, 1>(m, v, nullptr, m->ws.ug + m->E * 5 * NP, m->ws.uf + m->E * 30 * NF, s);
    return launch_interp64<N>(m, v, nullptr, 1, s);
  } else {
    const size_t sm = Smem<N, 1, R>::interp;
    int rc = set_smem(k_interp<N, 1, R, CM_NATIVE>, sm);
    if (rc) return rc;
    const unsigned blocks = (unsigned)((m->E + EPB - 1) / EPB);
    const WorkT<R> w = work_of<R>(m);
    prof_begin(m, s, KK_INTERP);
    k_interp<N, 1, R, CM_NATIVE><<<blocks, EPB * NP, sm, s>>>(v, nullptr, m->E, m->d_ops, w.ug + m->E * 5 * NP,
                                                               w.uf + m->E * 30 * NF);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_interp(tangent)");
    return DG_OK;
  }
}

template <int N, int NC, typename R = double>
static int run_faces(dg_mesh* m, cudaStream_t s, bool vout = true) {
  constexpr int NF = Shape<N>::NF;
  const long long work = m->nfaces * NF;
  // FP64: small CTAs, whose last wave leaves fewer SMs idle (one warp while the faces cannot fill every SM;
  // an 8x8x6 degree-2 stage solve 88.7 -> 80 ms against CTAs of 128)
  const int threads = !std::is_same<R, double>::value ? 128 : work <= NUM_SMS * 512 ? 32 : 64;
  const unsigned blocks = (unsigned)((work + threads - 1) / threads);
  const WorkT<R> w = work_of<R>(m);
  prof_begin(m, s, KK_FACES);
  if constexpr (std::is_same<R, double>::value)
    k_faces64<N, NC><<<blocks, threads, 0, s>>>(m->E, m->nfaces, phys_as<R>(m->phys), m->face_e, m->face_f, m->nbr,
                                                     m->nbr_fo, m->fgu, w.uf, w.qf, w.fh, w.mixf);
  else
    k_faces<N, NC, R><<<blocks, threads, 0, s>>>(m->E, m->nfaces, phys_as<R>(m->phys), m->face_e, m->face_f,
                                                       m->nbr, m->nbr_fo, w.fgeo, w.uf, w.qf, w.fh, w.mixf, vout);
  prof_end(m, s);
  DG_LAUNCH_CHECK("k_faces");
  return DG_OK;
}

// resident CTAs of kernel fn on the mesh's device at this launch shape (0 if the query fails),
// cached in the mesh
inline long long resident_ctas(dg_mesh* m, const void* fn, int threads, size_t smem) {
  OccCache& c = m->occ;
  for (int i = 0; i < c.n; ++i)
    if (c.fn[i] == fn && c.smem[i] == smem) return c.val[i];
  int per_sm = 0, sms = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device) != cudaSuccess) {
    cudaGetLastError();
    per_sm = sms = 0;
  }
  const long long v = (long long)per_sm * sms;
  if (c.n < OccCache::CAP) {
    c.fn[c.n] = fn;
    c.smem[c.n] = smem;
    c.val[c.n] = v;
    c.n++;
  }
  return v;
}

// the Sun of the heating models at time t
static Sun64 sun_at(const dg_mesh* m, double t) {
  Sun64 sun{{0.0, 0.0, 0.0}, m->d_euv};
  const double wt = m->phys.euv_omega_t * t;
  if (m->phys.euv == DG_EUV_GAUSS) {
    sun.d[0] = std::cos(wt);
    sun.d[1] = -std::sin(wt);
  } else if (m->phys.euv == DG_EUV_EUVAC) {
    sun.d[0] = -m->phys.sun_cd * std::cos(wt);
    sun.d[1] = m->phys.sun_cd * std::sin(wt);
    sun.d[2] = m->phys.sun_sd;
  }
  return sun;
}

template <int N, int NC, typename R = double, int CM = CM_NATIVE>
static int run_volume(dg_mesh* m, double t, double* r, double* jv, cudaStream_t s, double stage_c = 0.0) {
  if constexpr (std::is_same<R, double>::value) {
    using G = Grp<N>;
    const int threads = threads64<N>(m->E), per = threads / G::T;
    const size_t sm = sizeof(cell) * VolCells<N, NC>::size * per;
    int rc = set_smem(k_volume64<N, NC>, sizeof(cell) * VolCells<N, NC>::size * groups64_max<N>());
    if (rc) return rc;
    const Sun64 sun = sun_at(m, t);
    prof_begin(m, s, KK_VOLUME);
    k_volume64<N, NC><<<(unsigned)((m->E + per - 1) / per), threads, sm, s>>>(
        m->E, m->d_ops, phys_as<double>(m->phys), sun, m->gu, m->acc, m->xg, m->ws.ug, m->ws.qg, m->ws.fh, r, jv, stage_c,
        stage_c != 0.0 ? 1.0 / stage_c : 0.0, m->mixg);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_volume64");
    return DG_OK;
  } else {
    constexpr int EPB = Epb<N, NC>::value, NP = Shape<N>::NP;
    auto launch = [&](auto planes) {
      constexpr int OUT = decltype(planes)::value;
      const size_t sm = Smem<N, NC, R>::volume * OUT;
      const int rc = set_smem(k_volume<N, NC, OUT, R, CM>, sm);
      if (rc) return rc;
      const unsigned blocks = (unsigned)((m->E + EPB - 1) / EPB);
      const WorkT<R> w = work_of<R>(m);
      // CTAs resident at once (the prefetch distance), per mesh and kernel instance
      const long long resident = resident_ctas(m, (const void*)k_volume<N, NC, OUT, R, CM>, EPB * NP, sm);
      prof_begin(m, s, KK_VOLUME);
      k_volume<N, NC, OUT, R, CM><<<blocks, EPB * NP, sm, s>>>(m->E, m->d_ops, phys_as<R>(m->phys), (R)t, w.geo, w.acc,
                                                               w.xg, w.ug, w.qg, w.fh, r, jv, (R)stage_c, w.mixg, resident);
      prof_end(m, s);
      return (int)DG_OK;
    };
    const int rc = NC == 2 && !r ? launch(std::integral_constant<int, 1>()) : launch(std::integral_constant<int, NC>());
    if (rc) return rc;
    DG_LAUNCH_CHECK("k_volume");
    return DG_OK;
  }
}

template <int N>
int Driver<N>::cross_kappa(dg_mesh* m, double* kn) {
  constexpr int NF = Shape<N>::NF;
  k_cross_kappa<N><<<(unsigned)((m->E * 6 * NF + 127) / 128), 128>>>(m->E, m->d_ops, m->geo, m->fgeo, kn);
  DG_LAUNCH_CHECK("k_cross_kappa");
  return DG_OK;
}

template <int N>
int Driver<N>::geometry(dg_mesh* m, cudaStream_t s) {
  constexpr int NP = Shape<N>::NP;
  const size_t sm = sizeof(double) * 15 * NP;
  int rc = set_smem(k_geometry<N, false>, sm);
  if (rc == DG_OK) rc = set_smem(k_geometry<N, true>, sm);
  if (rc) return rc;
  const dg_mesh_desc& d = m->desc;
  prof_begin(m, s, KK_GEOMETRY);
  for (int unw = 0; unw < 2; ++unw) {
    auto kern = unw ? k_geometry<N, true> : k_geometry<N, false>;
    kern<<<(unsigned)m->E, NP < 32 ? 32 : NP, sm, s>>>(m->E, unw ? m->d_ops : m->d_ops_geo, m->phys, d.gravity_kind,
                                                      d.gvec[0], d.gvec[1], d.gvec[2], d.g_r0, m->x, m->geo, m->acc,
                                                      m->xg, m->fgeo, m->gu, m->fgu);
  }
  prof_end(m, s);
  DG_LAUNCH_CHECK("k_geometry");
  return DG_OK;
}

template <int N>
template <typename R>
int Driver<N>::gradient_p(dg_mesh* m, const double* u, const double* v, cudaStream_t s, bool tangent_only) {
  if (tangent_only) {   // u's value plane is in place: the tangent of v alone
    int rc = run_interp_tangent<N, R>(m, v, s);
    if (rc) return rc;
    return run_grad<N, 1, R, CM_NATIVE, true>(m, s);
  }
  int rc = v ? run_interp<N, 2, R>(m, u, v, s) : run_interp<N, 1, R>(m, u, nullptr, s);
  if (rc) return rc;
  return v ? run_grad<N, 2, R>(m, s) : run_grad<N, 1, R>(m, s);
}

template <int N>
template <typename R>
int Driver<N>::residual_p(dg_mesh* m, double t, double* r, double* jv, bool tangent, cudaStream_t s,
                          double stage_c) {
  int rc = tangent ? run_faces<N, 2, R>(m, s, r != nullptr) : run_faces<N, 1, R>(m, s);
  if (rc) return rc;
  return tangent ? run_volume<N, 2, R>(m, t, r, jv, s, stage_c) : run_volume<N, 1, R>(m, t, r, nullptr, s);
}

template <int N>
int Driver<N>::gradient(dg_mesh* m, const double* u, const double* v, cudaStream_t s, bool f32, bool tangent_only) {
  return f32 ? gradient_p<float>(m, u, v, s, tangent_only) : gradient_p<double>(m, u, v, s, tangent_only);
}

template <int N>
int Driver<N>::residual(dg_mesh* m, const double* u, const double* v, double t, double* r, double* jv,
                        bool tangent, cudaStream_t s, bool f32, double stage_c) {
  (void)u;
  (void)v;
  return f32 ? residual_p<float>(m, t, r, jv, tangent, s, stage_c)
             : residual_p<double>(m, t, r, jv, tangent, s, stage_c);
}

// the diagonal blocks of J_G = M - c J_r at the state whose value plane is in place; jac holds `batch`
// elements' Jacobians
template <int N>
int Driver<N>::blocks(dg_mesh* m, double t, double c, double* jac, long long batch, float* out, cudaStream_t s) {
  using B = Blk<N>;
  constexpr int NP = B::NP, NF = B::NF;
  const size_t sm = sizeof(cell) * B::cells;
  int rc = set_smem(k_blocks<N>, sm);
  if (rc) return rc;
  if (std::fabs(c) < STAGE_C_MIN) c = 0.0;   // M alone, to FP32's rounding for every |J_r| below 1e190 |M|
  const Sun64 sun = sun_at(m, t);
  const PhysT<double> P = phys_as<double>(m->phys);
  for (long long e0 = 0; e0 < m->E; e0 += batch) {
    const long long nE = m->E - e0 < batch ? m->E - e0 : batch;
    double* JF = jac + nE * B::JV;
    prof_begin(m, s, KK_VOLUME);
    k_jac_volume<N><<<(unsigned)((nE * NP + 127) / 128), 128, 0, s>>>(e0, nE, m->E, P, sun, m->gu, m->acc, m->xg, m->ws.ug,
                                                                    m->ws.qg, m->mixg, jac);
    prof_end(m, s);
    prof_begin(m, s, KK_FACES);
    k_jac_faces<N><<<(unsigned)((nE * 6 * NF + 127) / 128), 128, 0, s>>>(e0, nE, P, m->nbr, m->nbr_fo, m->fgu, m->kn,
                                                                       m->ws.uf, m->ws.qf, m->mixf, JF);
    prof_end(m, s);
    prof_begin(m, s, KK_LU);
    k_blocks<N><<<(unsigned)nE, B::GP * B::T, sm, s>>>(e0, m->d_ops, P.t_wall, m->gu, m->fgu, m->nbr, m->ws.uf, jac, JF,
                                                     c != 0.0 ? c : -1.0, c != 0.0, out);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_blocks");
  }
  return DG_OK;
}
// the same in FP32 at the state whose FP32 value plane is in place; jac holds `batch` elements' FP32 Jacobians
template <int N>
int Driver<N>::blocks_f32(dg_mesh* m, double t, double c, float* jac, long long batch, float* out, cudaStream_t s) {
  using B = Blk32<N>;
  constexpr int NP = B::NP, NF = B::NF;
  const size_t sm = sizeof(float) * B::floats;
  int rc = set_smem(k_blocks32<N>, sm);
  if (rc) return rc;
  const PhysT<float> P = phys_as<float>(m->phys);
  const WorkT<float> w = m->w32;
  for (long long e0 = 0; e0 < m->E; e0 += batch) {
    const long long nE = m->E - e0 < batch ? m->E - e0 : batch;
    float* JF = jac + nE * Blk<N>::JV;
    prof_begin(m, s, KK_VOLUME);
    k_jac_volume32<N><<<(unsigned)((nE * NP + 127) / 128), 128, 0, s>>>(e0, nE, P, (float)t, w.geo, w.acc, w.xg, w.ug, w.qg,
                                                                      w.mixg, jac);
    prof_end(m, s);
    prof_begin(m, s, KK_FACES);
    k_jac_faces32<N><<<(unsigned)((nE * 6 * NF + 127) / 128), 128, 0, s>>>(e0, nE, P, m->nbr, m->nbr_fo, w.fgeo, m->kn, w.uf,
                                                                         w.qf, w.mixf, JF);
    prof_end(m, s);
    prof_begin(m, s, KK_LU);
    k_blocks32<N><<<(unsigned)nE, B::GP * B::T, sm, s>>>(e0, m->d_ops, P.t_wall, w.geo, w.fgeo, m->nbr, w.uf, jac, JF,
                                                       (float)c, out);
    prof_end(m, s);
    DG_LAUNCH_CHECK("k_blocks32");
  }
  return DG_OK;
}
template <int N>
long long Driver<N>::block_doubles() { return Blk<N>::JV + Blk<N>::JF; }

template <int N>
template <int CM>
int Driver<N>::eval_cm_t(dg_mesh* m, const double* u, const double* v, double t, double* r, double* jv,
                         cudaStream_t s) {
  const bool tan = v != nullptr;
  int rc = tan ? run_interp<N, 2, float, CM>(m, u, v, s) : run_interp<N, 1, float, CM>(m, u, nullptr, s);
  if (rc) return rc;
  rc = tan ? run_grad<N, 2, float, CM>(m, s) : run_grad<N, 1, float, CM>(m, s);
  if (rc) return rc;
  rc = tan ? run_faces<N, 2, float>(m, s) : run_faces<N, 1, float>(m, s);
  if (rc) return rc;
  return tan ? run_volume<N, 2, float, CM>(m, t, r, jv, s) : run_volume<N, 1, float, CM>(m, t, r, nullptr, s);
}

template <int N>
int Driver<N>::eval_cm(dg_mesh* m, const double* u, const double* v, double t, double* r, double* jv, int cm,
                       cudaStream_t s) {
  switch (cm) {
    case CM_NATIVE: return eval_cm_t<CM_NATIVE>(m, u, v, t, r, jv, s);
    case CM_BF16: return eval_cm_t<CM_BF16>(m, u, v, t, r, jv, s);
    case CM_FP16: return eval_cm_t<CM_FP16>(m, u, v, t, r, jv, s);
    case CM_BF16X3: return eval_cm_t<CM_BF16X3>(m, u, v, t, r, jv, s);
    case CM_FP16X3: return eval_cm_t<CM_FP16X3>(m, u, v, t, r, jv, s);
    default: return fail(DG_EINVAL, "unknown contraction mode");
  }
}

template <int N, int MODE>
static int run_nodal(dg_mesh* m, const double* in, double* out, cudaStream_t s) {
  using G = Grp<N>;
  constexpr int planes = MODE == NODAL_FROM_GAUSS ? 3 : 1;
  const int threads = threads64<N>(m->E * planes), per = threads / G::T;
  const size_t sm = sizeof(cell) * 10 * G::NP * per;
  int rc = set_smem(k_nodal64<N, MODE>, sizeof(cell) * 10 * G::NP * groups64_max<N>());
  if (rc) return rc;
  prof_begin(m, s, KK_TENSOR);
  k_nodal64<N, MODE><<<dim3((unsigned)((m->E + per - 1) / per), planes), threads, sm, s>>>(m->E, m->d_ops, in, out, m->gu);
  prof_end(m, s);
  DG_LAUNCH_CHECK("k_nodal64");
  return DG_OK;
}

template <int N>
int Driver<N>::q_to_nodal(dg_mesh* m, double* q, cudaStream_t s) {
  return run_nodal<N, NODAL_FROM_GAUSS>(m, m->ws.qg, q, s);
}

template <int N>
int Driver<N>::q_from_nodal(dg_mesh* m, const double* q, cudaStream_t s) {
  using G = Grp<N>;
  const int threads = threads64<N>(m->E * 3), per = threads / G::T;
  const size_t sm = sizeof(cell) * 10 * G::NP * per;
  int rc = set_smem(k_interp64<N, true>, sizeof(cell) * 10 * G::NP * groups64_max<N>());
  if (rc) return rc;
  prof_begin(m, s, KK_TENSOR);
  k_interp64<N, true><<<dim3((unsigned)((m->E + per - 1) / per), 3), threads, sm, s>>>(q, nullptr, m->E, m->d_ops,
                                                                                     m->ws.qg, m->ws.qf);
  prof_end(m, s);
  DG_LAUNCH_CHECK("k_interp64(q)");
  return DG_OK;
}

template <int N>
int Driver<N>::mixture(dg_mesh* m) {
  k_mixture<N><<<(unsigned)m->E, 128>>>(m->E, m->d_ops_geo, m->phys, m->xg, m->mixg, m->mixf);
  DG_LAUNCH_CHECK("k_mixture");
  return DG_OK;
}

template <int N>
int Driver<N>::mass_inv(dg_mesh* m, const double* v, double* mv, cudaStream_t s) {
  return run_nodal<N, NODAL_MASS_INV>(m, v, mv, s);
}

template <int N>
int Driver<N>::mass(dg_mesh* m, const double* v, double* mv, cudaStream_t s) {
  return run_nodal<N, NODAL_MASS>(m, v, mv, s);
}

}  // namespace dg
