// Learned element preconditioner: features, network forward/backward, training and application.
//
// The paper has no learned component; this is the library's learned right preconditioner for
// the GMRES of Sec. 3.2. Per element e, with S_e the diagonal of the element mass matrix (one
// value per node, shared by the five variables) and Bs_e = S^{-1/2} B_e S^{-1/2} the scaled exact
// diagonal block of J_G, a two-hidden-layer SiLU network maps features x_e to
// D = 1 + o[:n], U = o[n : n + n r], V = o[n + n r :] (row-major n x r) and the preconditioner is
// P_e = S^{-1/2} (diag(D) + U V^T) S^{-1/2}. Training minimises
// L = mean_b || Bs_b (diag(D) + U V^T) - I ||_F^2 / n with Adam; the gradients are written out by
// hand (GEMM kernels for the layers, one CTA per sample for the loss). The loss measures P as a
// RIGHT inverse (|| Bs P - I ||) because GMRES applies it on the right.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "dg_internal.cuh"

namespace dg {

// ------------------------------------------------------------------------------------------
// FP32 tiled GEMM: C[m][n] = sum_k A(m,k) B(k,n)
// A(m,k) = TA ? A[k lda + m] : A[m lda + k];  B(k,n) = TB ? B[n ldb + k] : B[k ldb + n]
// The layers are small (a few hundred outputs each way), so K is split over grid.z until every SM has
// work: dh2 = dout W3 (512 x 256 outputs, K = 4455) took 1.04 ms on 32 CTAs. A split writes partial sums
// [z][M][N], which k_gemm_finish adds in order with the layer's epilogue. The forward layers (K of a few
// hundred) are not split: every element's outputs are the same whatever the number of rows. The next
// tile's global loads are in flight while the current one is multiplied (4 x 4 per thread, 16-byte shared
// loads).
// ------------------------------------------------------------------------------------------
constexpr int GBM = 64, GBN = 64, GBK = 16;

// v (+ bias); times silu'(z) when backward; *h = silu(v) when forward
__device__ __forceinline__ float gemm_epilogue(float v, const float* bias, int column, const float* Z, long long i, float* H) {
  if (bias) v += bias[column];
  if (Z) {
    const float sg = 1.f / (1.f + expf(-Z[i]));
    v *= sg * (1.f + Z[i] * (1.f - sg));
  }
  if (H) H[i] = v / (1.f + expf(-v));
  return v;
}

template <bool TA, bool TB>
__global__ void __launch_bounds__(256) k_gemm(int M, int N, int K, int kc, const float* __restrict__ A, int lda,
                                              const float* __restrict__ B, int ldb, float* __restrict__ C,
                                              const float* __restrict__ bias, float* __restrict__ H,
                                              const float* __restrict__ Z) {
  __shared__ __align__(16) float As[2][GBK][GBM + 4];
  __shared__ __align__(16) float Bs[2][GBK][GBN + 4];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int m0 = blockIdx.y * GBM, n0 = blockIdx.x * GBN;
  const int kb = blockIdx.z * kc, ke = min(K, kb + kc);
  float acc[4][4] = {};
  float ra[4], rb[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = tid + 256 * q;
      const int am = TA ? t % GBM : t / GBK, ak = k0 + (TA ? t / GBM : t % GBK);
      const int bn = TB ? t / GBK : t % GBN, bk = k0 + (TB ? t % GBK : t / GBN);
      ra[q] = (m0 + am < M && ak < ke) ? (TA ? A[(long long)ak * lda + m0 + am] : A[(long long)(m0 + am) * lda + ak]) : 0.f;
      rb[q] = (n0 + bn < N && bk < ke) ? (TB ? B[(long long)(n0 + bn) * ldb + bk] : B[(long long)bk * ldb + n0 + bn]) : 0.f;
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int t = tid + 256 * q;
      As[buf][TA ? t / GBM : t % GBK][TA ? t % GBM : t / GBK] = ra[q];
      Bs[buf][TB ? t % GBK : t / GBN][TB ? t / GBK : t % GBN] = rb[q];
    }
  };
  fetch(kb);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += GBK) {
    const bool more = k0 + GBK < ke;
    if (more) fetch(k0 + GBK);
#pragma unroll
    for (int kk = 0; kk < GBK; ++kk) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4]);
      const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][tx * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) stage(buf ^ 1);                // the other buffer: its readers passed the last barrier
    __syncthreads();
    buf ^= 1;
  }
  float* out = C + (long long)blockIdx.z * M * N;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gm = m0 + ty * 4 + i, gn = n0 + tx * 4 + j;
      if (gm < M && gn < N) {
        const long long at = (long long)gm * N + gn;
        out[at] = gridDim.z == 1 ? gemm_epilogue(acc[i][j], bias, gn, Z, at, H) : acc[i][j];
      }
    }
}

// C = sum_z part[z], then the epilogue
__global__ void k_gemm_finish(long long total, int N, int splits, const float* __restrict__ part, float* __restrict__ C,
                              const float* __restrict__ bias, float* __restrict__ H, const float* __restrict__ Z) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    float v = part[i];
    for (int z = 1; z < splits; ++z) v += part[z * total + i];
    C[i] = gemm_epilogue(v, bias, (int)(i % N), Z, i, H);
  }
}

// splits of K: enough for one CTA per SM, each with at least four K tiles
static int gemm_splits(int M, int N, int K) {
  const int tiles = ((N + GBN - 1) / GBN) * ((M + GBM - 1) / GBM);
  return std::max(1, std::min((NUM_SMS + tiles - 1) / tiles, K / (4 * GBK)));
}
static size_t gemm_part_floats(int M, int N, int K) {
  const int sp = gemm_splits(M, N, K);
  return sp > 1 ? (size_t)sp * M * N : 0;
}

template <bool TA, bool TB>
static void gemm(cudaStream_t s, int M, int N, int K, const float* A, int lda, const float* B, int ldb, float* C,
                 float* part, const float* bias = nullptr, float* H = nullptr, const float* Z = nullptr) {
  const int sp = part ? gemm_splits(M, N, K) : 1;   // part: room for gemm_part_floats, or no split
  const int kc = ((K + sp - 1) / sp + GBK - 1) / GBK * GBK;
  const int nz = (K + kc - 1) / kc;
  dim3 grid((N + GBN - 1) / GBN, (M + GBM - 1) / GBM, nz);
  k_gemm<TA, TB><<<grid, 256, 0, s>>>(M, N, K, kc, A, lda, B, ldb, nz > 1 ? part : C, bias, H, Z);
  const long long total = (long long)M * N;
  if (nz > 1) k_gemm_finish<<<(unsigned)std::min((total + 255) / 256, 1216LL), 256, 0, s>>>(total, N, nz, part, C, bias, H, Z);
}

// column sums of a [rows][cols] matrix (bias gradients), fixed order: 32 columns per CTA, rows over 16 warps
__global__ void __launch_bounds__(512) k_colsum(int rows, int cols, const float* __restrict__ X, float* __restrict__ out) {
  __shared__ float red[16][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * 32 + lane;
  float s = 0.f;
  if (c < cols)
    for (int r = warp; r < rows; r += 16) s += X[(long long)r * cols + c];
  red[warp][lane] = s;
  __syncthreads();
  if (warp == 0 && c < cols) {
    for (int w = 1; w < 16; ++w) s += red[w][lane];
    out[c] = s;
  }
}

// ------------------------------------------------------------------------------------------
// loss and output gradient, one CTA per sample, for P as a right inverse: R = Bs P - I, P = diag(D) + U V^T,
// G = scale Bs^T R:
//   W = Bs U (n x r);  R_ij = Bs_ij D_j + sum_k W_ik V_jk - delta_ij
//   dD_j = scale sum_i Bs_ij R_ij;  dV = scale R^T W;  Z = R V;  dU = scale Bs^T Z
// The block is read once, in strips of 16 rows held in shared memory: a strip gives its rows of W, R and Z
// and its share of the two transposed products, which stay in registers (4 x 4 tiles, NT per thread).
// 512 blocks of 135^2, rank 16: 1.15 ms with one row per thread and run-time indexed local arrays before.
// ------------------------------------------------------------------------------------------
constexpr int MLP_MAXR = 32;
constexpr int LG_RB = 16;
constexpr int LG_SMEM = 224 * 1024;

static size_t loss_smem(int n, int r) {
  const size_t r4 = (r + 3) / 4 * 4, n4 = (n + 3) / 4 * 4;
  return sizeof(float) * (2 * n4 * r4 + n4 + 2 * LG_RB * (n4 + 4) + LG_RB * 2 * r4 + 4096);
}

template <int NT>
__global__ void __launch_bounds__(256) k_loss_grad(int n, int r, const float* __restrict__ out,
                                                   const float* __restrict__ Bs, float scale, float* __restrict__ dout,
                                                   double* __restrict__ loss_part) {
  constexpr int RB = LG_RB;
  extern __shared__ __align__(16) float sm[];
  const int b = blockIdx.x, tid = threadIdx.x;
  const int no = n + 2 * n * r;
  const int r4 = (r + 3) / 4 * 4, n4 = (n + 3) / 4 * 4, C = 2 * r4, ldb = n4 + 4;
  const float* o = out + (long long)b * no;
  const float* Bm = Bs + (long long)b * n * n;       // row-major
  float* U = sm;                                     // [n4][r4], zero padded
  float* V = U + n4 * r4;                            // [n4][r4]
  float* D = V + n4 * r4;                            // [n4]
  float* Bb = D + n4;                                // [RB][ldb] rows of Bs
  float* Rb = Bb + RB * ldb;                         // [RB][ldb] rows of R
  float* Y = Rb + RB * ldb;                          // [RB][C]: W | Z
  float* red = Y + RB * C;                           // [4096]
  __shared__ double lred[256];
  for (int i = tid; i < n4; i += 256) D[i] = i < n ? 1.f + o[i] : 0.f;
  for (int i = tid; i < n4 * r4; i += 256) {
    const int j = i / r4, k = i % r4;
    const bool in = j < n && k < r;
    U[i] = in ? o[n + j * r + k] : 0.f;
    V[i] = in ? o[n + n * r + j * r + k] : 0.f;
  }
  // Y[:, c0 ...] = A (rows of a strip, n wide) times X [n][r4]: 4 x 4 tiles, n split over the other threads
  auto strip_times = [&](const float* A, const float* X, int c_out) {
    const int tiles = r4, KS = 256 / tiles;
    const int tile = tid % tiles, ks = tid / tiles;
    const int i0 = tile / (r4 / 4) * 4, c0 = tile % (r4 / 4) * 4;
    if (ks < KS) {
      float acc[4][4] = {};
      for (int j = ks; j < n; j += KS) {
        const float4 x = *reinterpret_cast<const float4*>(X + j * r4 + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float a = A[(i0 + q) * ldb + j];
          acc[q][0] = fmaf(a, x.x, acc[q][0]);
          acc[q][1] = fmaf(a, x.y, acc[q][1]);
          acc[q][2] = fmaf(a, x.z, acc[q][2]);
          acc[q][3] = fmaf(a, x.w, acc[q][3]);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int c = 0; c < 4; ++c) red[ks * (RB * r4) + (i0 + q) * r4 + c0 + c] = acc[q][c];
    }
    __syncthreads();
    for (int i = tid; i < RB * r4; i += 256) {
      float v = red[i];
      for (int q = 1; q < KS; ++q) v += red[q * (RB * r4) + i];
      Y[i / r4 * C + c_out + i % r4] = v;
    }
    __syncthreads();
  };
  float acc[NT][4][4] = {};
  float dd[2] = {0.f, 0.f};                          // columns tid, tid + 256
  double ls = 0.0;                                   // in FP64: squares beyond the FP32 range stay finite
  const int tiles2 = (n4 / 4) * (C / 4);
  for (int i0 = 0; i0 < n; i0 += RB) {
    __syncthreads();
    for (int i = tid; i < RB * n4; i += 256) {
      const int q = i / n4, j = i % n4;
      Bb[q * ldb + j] = (i0 + q < n && j < n) ? Bm[(long long)(i0 + q) * n + j] : 0.f;
    }
    __syncthreads();
    strip_times(Bb, U, 0);                           // W
#pragma unroll
    for (int h = 0; h < 2; ++h) {                    // R, the loss and dD: one column per thread
      const int j = tid + 256 * h;
      if (j >= n4) continue;
      float x[RB];
#pragma unroll
      for (int q = 0; q < RB; ++q) x[q] = Bb[q * ldb + j] * D[j] - (i0 + q == j ? 1.f : 0.f);
      for (int k = 0; k < r4; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(V + j * r4 + k);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
          const float4 w = *reinterpret_cast<const float4*>(Y + q * C + k);
          x[q] = fmaf(w.x, v.x, fmaf(w.y, v.y, fmaf(w.z, v.z, fmaf(w.w, v.w, x[q]))));
        }
      }
#pragma unroll
      for (int q = 0; q < RB; ++q) {
        if (i0 + q >= n || j >= n) x[q] = 0.f;
        Rb[q * ldb + j] = x[q];
        dd[h] = fmaf(Bb[q * ldb + j], x[q], dd[h]);
        const double xd = to_f64_exact(x[q]);
        ls = fma(xd, xd, ls);
      }
    }
    __syncthreads();
    strip_times(Rb, V, r4);                          // Z
#pragma unroll
    for (int h = 0; h < NT; ++h) {                   // R^T W and Bs^T Z
      const int tile = tid + 256 * h;
      if (tile >= tiles2) continue;
      const int j0 = tile % (n4 / 4) * 4, c0 = tile / (n4 / 4) * 4;
      const float* A = c0 < r4 ? Rb : Bb;
#pragma unroll 4
      for (int q = 0; q < RB; ++q) {
        const float4 a = *reinterpret_cast<const float4*>(A + q * ldb + j0);
        const float4 y = *reinterpret_cast<const float4*>(Y + q * C + c0);
        const float av[4] = {a.x, a.y, a.z, a.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int w = 0; w < 4; ++w) acc[h][u][w] = fmaf(av[u], yv[w], acc[h][u][w]);
      }
    }
  }
  float* g = dout + (long long)b * no;
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (tid + 256 * h < n) g[tid + 256 * h] = scale * dd[h];
#pragma unroll
  for (int h = 0; h < NT; ++h) {
    const int tile = tid + 256 * h;
    if (tile >= tiles2) continue;
    const int j0 = tile % (n4 / 4) * 4, c0 = tile / (n4 / 4) * 4;
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        const int j = j0 + u, k = c0 < r4 ? c0 + w : c0 - r4 + w;
        if (j < n && k < r) g[n + (c0 < r4 ? n * r : 0) + j * r + k] = scale * acc[h][u][w];
      }
  }
  lred[tid] = ls;
  __syncthreads();
  for (int st = 128; st > 0; st >>= 1) {
    if (tid < st) lred[tid] += lred[tid + st];
    __syncthreads();
  }
  if (tid == 0) loss_part[b] = lred[0];
}

static int launch_loss(int nb, int n, int r, const float* out, const float* Bs, float scale, float* dout,
                       double* loss_part, cudaStream_t s) {
  const size_t smem = loss_smem(n, r);
  const int r4 = (r + 3) / 4 * 4, n4 = (n + 3) / 4 * 4;
  const int nt = ((n4 / 4) * (2 * r4 / 4) + 255) / 256;
  if (smem > LG_SMEM || n > 512 || nt > 5) return fail(DG_EINVAL, "MLP block too large for the loss kernel");
  auto go = [&](auto kern) -> int {
    // the same limit for every network (threads may train others), beside the kernel's static 2 KB
    DG_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LG_SMEM));
    kern<<<nb, 256, smem, s>>>(n, r, out, Bs, scale, dout, loss_part);
    return DG_OK;
  };
  switch (nt) {
    case 1: return go(k_loss_grad<1>);
    case 2: return go(k_loss_grad<2>);
    case 3: return go(k_loss_grad<3>);
    case 4: return go(k_loss_grad<4>);
    default: return go(k_loss_grad<5>);
  }
}

__global__ void k_adam(long long n, float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// ------------------------------------------------------------------------------------------
// features and mass-diagonal scaling (one CTA per element, threads over nodes)
//   x = [varrho_i - mean, v_x, v_y, v_z, T_i / mean(T) - 1 (per node), mean(varrho)/10,
//        log mean(T), log(dt a_ii), log h_1, log h_2, log h_3]
//   S_i = sum_g (w |J|)_g phi_i(g)^2 (diagonal of the element mass matrix)
// ------------------------------------------------------------------------------------------
__global__ void k_features(long long E, int n, const double* __restrict__ u, const double* __restrict__ x,
                           const double* __restrict__ geo, const Ops* __restrict__ ops, double dt_aii,
                           float* __restrict__ feat, float* __restrict__ sdiag) {
  const int np = n * n * n;
  const long long e = blockIdx.x;
  const double* ue = u + e * 5 * np;
  const int nin = 5 * np + 6;
  float* f = feat + e * nin;
  __shared__ double s_r[256], s_t[256];
  double rsum = 0.0, tsum = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) {
    const double isr = exp(-0.5 * ue[i]);
    rsum += ue[i];
    tsum += ue[4 * np + i] * isr;
  }
  s_r[threadIdx.x] = rsum;
  s_t[threadIdx.x] = tsum;
  __syncthreads();
  for (int st = blockDim.x / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) {
      s_r[threadIdx.x] += s_r[threadIdx.x + st];
      s_t[threadIdx.x] += s_t[threadIdx.x + st];
    }
    __syncthreads();
  }
  const double rmean = s_r[0] / np, tmean = s_t[0] / np;
  for (int i = threadIdx.x; i < np; i += blockDim.x) {
    const double isr = exp(-0.5 * ue[i]);
    f[i] = (float)(ue[i] - rmean);
    f[np + i] = (float)(ue[np + i] * isr);
    f[2 * np + i] = (float)(ue[2 * np + i] * isr);
    f[3 * np + i] = (float)(ue[3 * np + i] * isr);
    f[4 * np + i] = (float)(ue[4 * np + i] * isr / tmean - 1.0);
    // mass diagonal: sum over Gauss points of w|J| phi_i^2, phi_i(g) = B[g1][a] B[g2][b] B[g3][c]
    const int a = i % n, bb = (i / n) % n, c = i / (n * n);
    double s = 0.0;
    for (int g = 0; g < np; ++g) {
      const int g1 = g % n, g2 = (g / n) % n, g3 = g / (n * n);
      const double ph = ops->B[g1 * n + a] * ops->B[g2 * n + bb] * ops->B[g3 * n + c];
      s += geo[e * 10 * np + 9 * np + g] * ph * ph;
    }
    sdiag[e * np + i] = (float)s;
  }
  if (threadIdx.x == 0) {
    const double* xe = x + e * 3 * np;
    f[5 * np] = (float)(rmean / 10.0);
    f[5 * np + 1] = (float)log(tmean);
    f[5 * np + 2] = (float)log(dt_aii);
    const int corner[3] = {n - 1, (n - 1) * n, (n - 1) * n * n};
    for (int d = 0; d < 3; ++d) {
      double h2 = 0.0;
      for (int k = 0; k < 3; ++k) {
        const double dx = xe[k * np + corner[d]] - xe[k * np];
        h2 += dx * dx;
      }
      f[5 * np + 3 + d] = (float)(0.5 * log(h2));
    }
  }
}

// Bs[e][i][j] = block[e][j][i] / sqrt(S_i S_j) (row-major), node of DOF i = i mod np
__global__ void k_scale_blocks(long long E, int np, const float* __restrict__ blocks, const float* __restrict__ sdiag,
                               float* __restrict__ Bs) {
  const int nb = 5 * np;
  const long long e = blockIdx.x;
  const float* Bc = blocks + e * (long long)nb * nb;
  float* Bo = Bs + e * (long long)nb * nb;
  for (int t = threadIdx.x; t < nb * nb; t += blockDim.x) {
    const int i = t / nb, j = t % nb;
    Bo[t] = Bc[(long long)j * nb + i] * rsqrtf(sdiag[e * np + i % np] * sdiag[e * np + j % np]);
  }
}

// y = S^{-1/2} (D * xs + U (V^T xs)), xs = S^{-1/2} x, per element (FP64 in and out)
__global__ void k_mlp_apply(long long E, int np, int r, const float* __restrict__ out, const float* __restrict__ sdiag,
                            const double* __restrict__ x, double* __restrict__ y) {
  extern __shared__ float sx[];
  __shared__ float tk[MLP_MAXR];
  const int nb = 5 * np, no = nb + 2 * nb * r;
  const long long e = blockIdx.x;
  const float* o = out + e * no;
  for (int i = threadIdx.x; i < nb; i += blockDim.x) sx[i] = (float)x[e * nb + i] * rsqrtf(sdiag[e * np + i % np]);
  __syncthreads();
  // t_k = sum_i V[i][k] xs_i: one warp per k
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32, nw = blockDim.x / 32;
  for (int k = warp; k < r; k += nw) {
    float acc = 0.f;
    for (int i = lane; i < nb; i += 32) acc = fmaf(o[nb + nb * r + i * r + k], sx[i], acc);
    for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
    if (lane == 0) tk[k] = acc;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += blockDim.x) {
    float v = (1.f + o[i]) * sx[i];
    for (int k = 0; k < r; ++k) v = fmaf(o[nb + i * r + k], tk[k], v);
    y[e * nb + i] = (double)(v * rsqrtf(sdiag[e * np + i % np]));
  }
}

// ------------------------------------------------------------------------------------------
// state
// ------------------------------------------------------------------------------------------
struct Mlp {
  int n_in = 0, hidden = 0, n = 0, rank = 0, n_out = 0;
  long long n_params = 0;
  float* params = nullptr;    // W1 b1 W2 b2 W3 b3
  float* grads = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  long long adam_t = 0;
  // training set
  long long cap = 0, count = 0;
  float* X = nullptr;         // [cap][n_in]
  float* Bs = nullptr;        // [cap][n][n]
  // scratch for a batch and for inference
  int batch_cap = 0;
  float *z1 = nullptr, *h1 = nullptr, *z2 = nullptr, *h2 = nullptr, *o = nullptr, *dout = nullptr, *dh = nullptr,
        *part = nullptr;
  double* loss_part = nullptr;
  // inference outputs for every element
  float* feat = nullptr;      // [E][n_in]
  float* sdiag = nullptr;     // [E][np]
  float* outE = nullptr;      // [E][n_out]
  bool ready = false;
  float* W1() { return params; }
  float* b1() { return W1() + (long long)hidden * n_in; }
  float* W2() { return b1() + hidden; }
  float* b2() { return W2() + (long long)hidden * hidden; }
  float* W3() { return b2() + hidden; }
  float* b3() { return W3() + (long long)n_out * hidden; }
};

static void mlp_free(Mlp* M) {
  if (!M) return;
  void* p[] = {M->params, M->grads, M->adam_m, M->adam_v, M->X, M->Bs, M->z1, M->h1, M->z2, M->h2, M->o, M->dout,
               M->dh, M->part, M->loss_part, M->feat, M->sdiag, M->outE};
  for (void* q : p)
    if (q) cudaFree(q);
  delete M;
}

// SplitMix64 (Steele, Lea & Flood 2014) for the initial weights
static inline uint64_t splitmix(uint64_t seed, uint64_t i) {
  uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ULL;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}

static int ensure_batch(Mlp* M, int batch) {
  if (M->batch_cap >= batch) return DG_OK;
  auto release = [&]() {                     // and no batch fits: a failed call leaves nothing half allocated
    float** bufs[] = {&M->z1, &M->h1, &M->z2, &M->h2, &M->o, &M->dout, &M->dh, &M->part};
    for (float** b : bufs)
      if (*b) { cudaFree(*b); *b = nullptr; }
    if (M->loss_part) cudaFree(M->loss_part);
    M->loss_part = nullptr;
    M->batch_cap = 0;
  };
  release();
  const size_t H = (size_t)batch * M->hidden, OB = (size_t)batch * M->n_out;
  cudaError_t err = cudaMalloc(&M->z1, H * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->h1, H * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->z2, H * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->h2, H * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->o, OB * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->dout, OB * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->dh, (H > (size_t)batch * M->n_in ? H : (size_t)batch * M->n_in) * 4);
  if (err == cudaSuccess) err = cudaMalloc(&M->loss_part, sizeof(double) * batch);
  // partial sums of the split products, for every batch up to this one: fewer rows may split more, no more than
  // NUM_SMS tiles of 64 rows at all
  const int Hd = M->hidden, O = M->n_out, I = M->n_in;
  size_t part = 1;
  for (long long rows = GBM; rows < (long long)batch + GBM && rows <= (NUM_SMS + 1) * GBM; rows += GBM) {
    const int nb = (int)std::min(rows, (long long)batch);
    part = std::max(part, std::max(gemm_part_floats(nb, Hd, Hd), gemm_part_floats(nb, Hd, O)));
  }
  for (size_t p : {gemm_part_floats(O, Hd, batch), gemm_part_floats(Hd, Hd, batch), gemm_part_floats(Hd, I, batch)})
    part = std::max(part, p);
  if (err == cudaSuccess) err = cudaMalloc(&M->part, part * 4);
  if (err != cudaSuccess) {
    release();
    return fail(DG_ENOMEM, std::string("MLP batch storage: ") + cudaGetErrorString(err));
  }
  M->batch_cap = batch;
  return DG_OK;
}

static int forward(Mlp* M, const float* X, int nb, float* out, cudaStream_t s) {
  gemm<false, true>(s, nb, M->hidden, M->n_in, X, M->n_in, M->W1(), M->n_in, M->z1, nullptr, M->b1(), M->h1);
  gemm<false, true>(s, nb, M->hidden, M->hidden, M->h1, M->hidden, M->W2(), M->hidden, M->z2, nullptr, M->b2(), M->h2);
  gemm<false, true>(s, nb, M->n_out, M->hidden, M->h2, M->hidden, M->W3(), M->hidden, out, nullptr, M->b3());
  DG_LAUNCH_CHECK("mlp forward");
  return DG_OK;
}

// loss over nb samples (X, Bs on the device) and parameter gradients into M->grads
static int loss_grad(Mlp* M, const float* X, const float* Bs, int nb, double* loss, cudaStream_t s) {
  int rc = ensure_batch(M, nb);
  if (rc) return rc;
  rc = forward(M, X, nb, M->o, s);
  if (rc) return rc;
  const float scale = 2.f / ((float)nb * (float)M->n);
  rc = launch_loss(nb, M->n, M->rank, M->o, Bs, scale, M->dout, M->loss_part, s);
  if (rc) return rc;
  DG_LAUNCH_CHECK("k_loss_grad");
  const int H = M->hidden, I = M->n_in, O = M->n_out;
  float* gW1 = M->grads;
  float* gb1 = gW1 + (long long)H * I;
  float* gW2 = gb1 + H;
  float* gb2 = gW2 + (long long)H * H;
  float* gW3 = gb2 + H;
  float* gb3 = gW3 + (long long)O * H;
  // output layer
  gemm<true, false>(s, O, H, nb, M->dout, O, M->h2, H, gW3, M->part);
  k_colsum<<<(O + 31) / 32, 512, 0, s>>>(nb, O, M->dout, gb3);
  // dz2 = (dout W3) silu'(z2)
  gemm<false, false>(s, nb, H, O, M->dout, O, M->W3(), H, M->dh, M->part, nullptr, nullptr, M->z2);
  gemm<true, false>(s, H, H, nb, M->dh, H, M->h1, H, gW2, M->part);
  k_colsum<<<(H + 31) / 32, 512, 0, s>>>(nb, H, M->dh, gb2);
  // dz1 = (dz2 W2) silu'(z1), into z2's buffer, no longer needed
  gemm<false, false>(s, nb, H, H, M->dh, H, M->W2(), H, M->z2, M->part, nullptr, nullptr, M->z1);
  gemm<true, false>(s, H, I, nb, M->z2, H, X, I, gW1, M->part);
  k_colsum<<<(H + 31) / 32, 512, 0, s>>>(nb, H, M->z2, gb1);
  DG_LAUNCH_CHECK("mlp backward");
  if (loss) {
    std::vector<double> part(nb);
    DG_CUDA_TRY(cudaMemcpyAsync(part.data(), M->loss_part, sizeof(double) * nb, cudaMemcpyDeviceToHost, s));
    DG_CUDA_TRY(cudaStreamSynchronize(s));
    double L = 0.0;
    for (double v : part) L += v;
    *loss = L / ((double)nb * M->n);
  }
  return DG_OK;
}

}  // namespace dg

void dg_mlp_release(dg_mesh* m) {
  dg::mlp_free(m->mlp);
  m->mlp = nullptr;
}

using namespace dg;

extern "C" int dg_mlp_init(dg_mesh* mesh, int32_t hidden, int32_t rank, int64_t max_samples, uint64_t seed) {
  if (!mesh || hidden < 1 || rank < 1 || rank > MLP_MAXR || max_samples < 0)
    return fail(DG_EINVAL, "dg_mlp_init: bad argument");
  if (mesh->n > 4) return fail(DG_EINVAL, "dg_mlp_init: the learned preconditioner supports p <= 3");
  dg_mlp_release(mesh);
  Mlp* M = new Mlp();
  M->n = 5 * mesh->np;
  M->n_in = 5 * mesh->np + 6;
  M->hidden = hidden;
  M->rank = rank;
  M->n_out = M->n + 2 * M->n * rank;
  M->n_params = (long long)hidden * M->n_in + hidden + (long long)hidden * hidden + hidden +
                (long long)M->n_out * hidden + M->n_out;
  M->cap = max_samples;
  const long long E = mesh->E;
  cudaError_t err = cudaMalloc(&M->params, sizeof(float) * M->n_params);
  if (err == cudaSuccess) err = cudaMalloc(&M->grads, sizeof(float) * M->n_params);
  if (err == cudaSuccess) err = cudaMalloc(&M->adam_m, sizeof(float) * M->n_params);
  if (err == cudaSuccess) err = cudaMalloc(&M->adam_v, sizeof(float) * M->n_params);
  if (err == cudaSuccess && max_samples) err = cudaMalloc(&M->X, sizeof(float) * max_samples * M->n_in);
  if (err == cudaSuccess && max_samples) err = cudaMalloc(&M->Bs, sizeof(float) * max_samples * M->n * M->n);
  if (err == cudaSuccess) err = cudaMalloc(&M->feat, sizeof(float) * E * M->n_in);
  if (err == cudaSuccess) err = cudaMalloc(&M->sdiag, sizeof(float) * E * mesh->np);
  if (err == cudaSuccess) err = cudaMalloc(&M->outE, sizeof(float) * E * M->n_out);
  if (err != cudaSuccess) {
    mlp_free(M);
    return fail(DG_ENOMEM, std::string("dg_mlp_init: ") + cudaGetErrorString(err));
  }
  // initial weights: uniform(-a, a), a = sqrt(6 / fan_in) for the hidden layers (SiLU), 0.1 of that
  // for the output layer, zero biases (the initial preconditioner is close to the mass scaling)
  std::vector<float> h(M->n_params, 0.f);
  long long off = 0, idx = 0;
  auto fill = [&](long long count, int fan_in, float gain) {
    const float a = gain * std::sqrt(6.f / (float)fan_in);
    for (long long k = 0; k < count; ++k) {
      const double u01 = (double)(splitmix(seed, (uint64_t)idx++) >> 11) * (1.0 / 9007199254740992.0);
      h[off + k] = (float)((2.0 * u01 - 1.0) * a);
    }
    off += count;
  };
  fill((long long)hidden * M->n_in, M->n_in, 1.f);
  off += hidden;
  fill((long long)hidden * hidden, hidden, 1.f);
  off += hidden;
  fill((long long)M->n_out * hidden, hidden, 0.1f);
  err = cudaMemcpy(M->params, h.data(), sizeof(float) * M->n_params, cudaMemcpyHostToDevice);
  if (err == cudaSuccess) err = cudaMemset(M->adam_m, 0, sizeof(float) * M->n_params);
  if (err == cudaSuccess) err = cudaMemset(M->adam_v, 0, sizeof(float) * M->n_params);
  if (err != cudaSuccess) {
    mlp_free(M);
    return fail(DG_ECUDA, std::string("dg_mlp_init: ") + cudaGetErrorString(err));
  }
  mesh->mlp = M;
  return DG_OK;
}

extern "C" int dg_mlp_sizes(dg_mesh* mesh, int64_t* n_params, int32_t* n_in, int32_t* n_out, int64_t* n_samples) {
  if (!mesh || !mesh->mlp) return fail(DG_EINVAL, "dg_mlp_sizes: no network");
  if (n_params) *n_params = mesh->mlp->n_params;
  if (n_in) *n_in = mesh->mlp->n_in;
  if (n_out) *n_out = mesh->mlp->n_out;
  if (n_samples) *n_samples = mesh->mlp->count;
  return DG_OK;
}

extern "C" int dg_mlp_params(dg_mesh* mesh, float* out, const float* in, void* stream) {
  if (!mesh || !mesh->mlp) return fail(DG_EINVAL, "dg_mlp_params: no network");
  Mlp* M = mesh->mlp;
  cudaStream_t s = (cudaStream_t)stream;
  if (out) DG_CUDA_TRY(cudaMemcpyAsync(out, M->params, sizeof(float) * M->n_params, cudaMemcpyDeviceToDevice, s));
  if (in) {
    DG_CUDA_TRY(cudaMemcpyAsync(M->params, in, sizeof(float) * M->n_params, cudaMemcpyDeviceToDevice, s));
    M->ready = false;
  }
  return DG_OK;
}

// features (and mass diagonal) of every element at state u
static int mlp_features(dg_mesh* mesh, const double* u, double dt_aii, cudaStream_t s) {
  Mlp* M = mesh->mlp;
  k_features<<<(unsigned)mesh->E, 128, 0, s>>>(mesh->E, mesh->n, u, mesh->x, mesh->geo, mesh->d_ops, dt_aii, M->feat,
                                               M->sdiag);
  DG_LAUNCH_CHECK("k_features");
  return DG_OK;
}

extern "C" int dg_mlp_features(dg_mesh* mesh, const double* u, double dt_aii, float* feat, float* sdiag, void* stream) {
  if (!mesh || !mesh->mlp || !u) return fail(DG_EINVAL, "dg_mlp_features: bad argument");
  cudaStream_t s = (cudaStream_t)stream;
  int rc = mlp_features(mesh, u, dt_aii, s);
  if (rc) return rc;
  Mlp* M = mesh->mlp;
  if (feat) DG_CUDA_TRY(cudaMemcpyAsync(feat, M->feat, sizeof(float) * mesh->E * M->n_in, cudaMemcpyDeviceToDevice, s));
  if (sdiag) DG_CUDA_TRY(cudaMemcpyAsync(sdiag, M->sdiag, sizeof(float) * mesh->E * mesh->np, cudaMemcpyDeviceToDevice, s));
  return DG_OK;
}

extern "C" int dg_mlp_harvest(dg_mesh* mesh, const double* u, double t, double dt_aii, int32_t stride,
                              int64_t* n_samples, void* stream) {
  if (!mesh || !mesh->mlp || !u || stride < 1) return fail(DG_EINVAL, "dg_mlp_harvest: bad argument");
  Mlp* M = mesh->mlp;
  cudaStream_t s = (cudaStream_t)stream;
  const long long E = mesh->E, nb = M->n;
  float* blocks = nullptr;
  DG_CUDA_TRY(cudaMalloc(&blocks, sizeof(float) * E * nb * nb));
  int rc = dg_block_assemble(mesh, u, t, dt_aii, blocks, stream);
  if (rc == DG_OK) rc = mlp_features(mesh, u, dt_aii, s);
  float* scaled = nullptr;
  if (rc == DG_OK && cudaMalloc(&scaled, sizeof(float) * E * nb * nb) != cudaSuccess) rc = fail(DG_ENOMEM, "harvest");
  if (rc == DG_OK) {
    k_scale_blocks<<<(unsigned)E, 256, 0, s>>>(E, mesh->np, blocks, M->sdiag, scaled);
    for (long long e = 0; e < E && M->count < M->cap; e += stride) {
      cudaMemcpyAsync(M->X + M->count * M->n_in, M->feat + e * M->n_in, sizeof(float) * M->n_in,
                      cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(M->Bs + M->count * nb * nb, scaled + e * nb * nb, sizeof(float) * nb * nb,
                      cudaMemcpyDeviceToDevice, s);
      M->count++;
    }
    cudaError_t err = cudaStreamSynchronize(s);
    if (err != cudaSuccess) rc = fail(DG_ECUDA, std::string("dg_mlp_harvest: ") + cudaGetErrorString(err));
  }
  cudaFree(blocks);
  if (scaled) cudaFree(scaled);
  if (n_samples) *n_samples = M->count;
  return rc;
}

extern "C" int dg_mlp_loss_grad(dg_mesh* mesh, const float* X, const float* Bs, int32_t nb, double* loss, float* grad,
                                void* stream) {
  if (!mesh || !mesh->mlp || !X || !Bs || nb < 1) return fail(DG_EINVAL, "dg_mlp_loss_grad: bad argument");
  Mlp* M = mesh->mlp;
  cudaStream_t s = (cudaStream_t)stream;
  int rc = loss_grad(M, X, Bs, nb, loss, s);
  if (rc) return rc;
  if (grad) DG_CUDA_TRY(cudaMemcpyAsync(grad, M->grads, sizeof(float) * M->n_params, cudaMemcpyDeviceToDevice, s));
  return DG_OK;
}

extern "C" int dg_mlp_train(dg_mesh* mesh, int32_t epochs, int32_t batch, double lr, double* loss_first,
                            double* loss_last, void* stream) {
  if (!mesh || !mesh->mlp || epochs < 1 || batch < 1) return fail(DG_EINVAL, "dg_mlp_train: bad argument");
  Mlp* M = mesh->mlp;
  if (M->count < 1) return fail(DG_EINVAL, "dg_mlp_train: no harvested samples");
  cudaStream_t s = (cudaStream_t)stream;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  double first = -1.0, last = 0.0;
  for (int ep = 0; ep < epochs; ++ep) {
    double esum = 0.0;
    long long seen = 0;
    for (long long off = 0; off < M->count; off += batch) {
      const int nb = (int)((M->count - off < batch) ? (M->count - off) : batch);
      double L = 0.0;
      const bool want = (off + batch >= M->count) || ep == 0;
      int rc = loss_grad(M, M->X + off * M->n_in, M->Bs + off * (long long)M->n * M->n, nb, want ? &L : nullptr, s);
      if (rc) return rc;
      ++M->adam_t;
      const float c1 = 1.f - std::pow(b1, (float)M->adam_t), c2 = 1.f - std::pow(b2, (float)M->adam_t);
      k_adam<<<1024, 256, 0, s>>>(M->n_params, M->params, M->grads, M->adam_m, M->adam_v, (float)lr, b1, b2, c1, c2,
                                  eps);
      DG_LAUNCH_CHECK("k_adam");
      if (want) {
        esum += L * nb;
        seen += nb;
      }
    }
    if (ep == 0 && seen) first = esum / seen;
    if (seen) last = esum / seen;
  }
  M->ready = false;
  if (loss_first) *loss_first = first;
  if (loss_last) *loss_last = last;
  return DG_OK;
}

// inference for every element at state u: stores D, U, V (scaled) for dg_precond_apply
int mlp_setup(dg_mesh* mesh, const double* u, double dt_aii, cudaStream_t s) {
  Mlp* M = mesh->mlp;
  if (!M) return fail(DG_EINVAL, "learned preconditioner used before dg_mlp_init");
  int rc = mlp_features(mesh, u, dt_aii, s);
  if (rc) return rc;
  const int chunk = 8192;
  rc = ensure_batch(M, chunk);
  if (rc) return rc;
  for (long long e0 = 0; e0 < mesh->E; e0 += chunk) {
    const int nb = (int)((mesh->E - e0 < chunk) ? mesh->E - e0 : chunk);
    rc = forward(M, M->feat + e0 * M->n_in, nb, M->outE + e0 * M->n_out, s);
    if (rc) return rc;
  }
  M->ready = true;
  return DG_OK;
}

int mlp_apply(dg_mesh* mesh, const double* x, double* y, cudaStream_t s) {
  Mlp* M = mesh->mlp;
  if (!M || !M->ready) return fail(DG_EINVAL, "learned preconditioner used before dg_precond_setup");
  k_mlp_apply<<<(unsigned)mesh->E, 128, sizeof(float) * M->n, s>>>(mesh->E, mesh->np, M->rank, M->outE, M->sdiag, x, y);
  DG_LAUNCH_CHECK("k_mlp_apply");
  return DG_OK;
}
