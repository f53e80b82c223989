// Small dense linear algebra of a split whose sketch is wider than one CTA's shared memory (k + p above 72, up to
// 272: the rank-128 and rank-256 points of the 70B-shaped sweep).  Same steps as the one-CTA kernels of split.cu
// (Section 3.1: thin QR of the sketch, small SVD of the projected operand), as kernels that tile over the rank:
//
//   gram64_kernel            G = V^T V in FP64, 64 x 64 output tiles over slabs of rows (partials, summed in order)
//   chol_mid_kernel          Cholesky factor of a q x q Gram matrix and the inverses of its diagonal blocks, one CTA: q up to
//                            160, the matrix in shared memory
//   chol_wide_kernel         the same above that: panels of 32 columns in shared memory, the matrix in L2
//   trsm_wide_kernel         H = Z L^-T by blocked forward substitution (32 rows of Z per CTA, FP64 tensor cores)
//   gemm64_kernel            C = A B with FP32 A, FP64 B and FP64 accumulation, arbitrary strides (right basis,
//                            factor rotations)
//   tridiag_chol_kernel      up to 144: Householder reduction in one CTA's registers beside the factorisation in another's shared
//                            memory; tridiag_vectors_kernel, tridiag_back_kernel: eigenvectors of the tridiagonal matrix, taken back
//   jacobi_fp32_kernel       above that, FP32 one-sided block Jacobi on a cluster of four to six CTAs: the columns live in the
//                            cluster's distributed shared memory, column blocks travel between CTAs by DSMEM stores
//   refine_*_kernel          FP64 refinement of the eigenvectors they found (steps of matrix products), eigen_finish_kernel
//   jacobi_cluster_kernel    the FP64 form of the sweeps, and jacobi_collect_kernel: only run for matrices the refinement
//                            cannot finish (eigenvalues that agree to working precision)
//   sign_rows_kernel         sign convention of the factor pairs
//   coef_sum_kernel          sums the column slices of the broadcast pass into a group of coefficient columns
// Included by split.cu only.
#pragma once
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"
#include "small_eig.cuh"

namespace metis_wide {

namespace cg = cooperative_groups;

constexpr int MAXQ_WIDE = 272;                          // 2 * JC_P * JC_W
constexpr int MAXK_WIDE = 256;

// ------------------------------------------------------------------------------------------------
// part[p][i][j] = sum over the p-th slab of rows r of v(r, i) v(r, j),  v(r, i) = V[r * sr + i * sv], FP64.
// grid (tiles_j, tiles_i, slabs).
// On the FP64 tensor cores: a warp owns 16 x 32 of the tile; tiles above the diagonal are the mirror image of those below it
// (as FP64 multiply-adds from shared memory over all tiles a rank-128 step spent 305 us on it, 190 us so).
constexpr int G64_T = 64, G64_R = 32, G64_P = G64_T + 4;
// acc (this warp's 16 x 32 of a 64 x 64 tile) += sum over kk < G64_R of as[kk][.] bs[kk][.]
__device__ __forceinline__ void tile64_mac(const double (*as)[G64_P], const double (*bs)[G64_P], int wm, int wn, int g, int q, double (&acc)[2][4][2]) {
#pragma unroll
  for (int kk = 0; kk < G64_R; kk += 4) {
    double a[2], b[4];
#pragma unroll
    for (int u = 0; u < 2; ++u) a[u] = as[kk + q][wm + 8 * u + g];
#pragma unroll
    for (int u = 0; u < 4; ++u) b[u] = bs[kk + q][wn + 8 * u + g];
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) metis_small::dmma(acc[u][v], a[u], b[v]);
  }
}
__global__ void __launch_bounds__(256)
gram64_kernel(const float* __restrict__ v, int64_t n_rows, int n, int64_t sr, int64_t sv, int64_t rows_per_part,
              double* __restrict__ part, const int* __restrict__ skip) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double as[G64_R][G64_P], bs[G64_R][G64_P];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, wm = 16 * (warp & 3), wn = 32 * (warp >> 2);
  const int i0 = blockIdx.y * G64_T, j0 = blockIdx.x * G64_T;
  const int64_t r_begin = (int64_t)blockIdx.z * rows_per_part, r_end = min(n_rows, r_begin + rows_per_part);
  double acc[2][4][2] = {};
  constexpr int PER = G64_R * G64_T / 256;                // values of either operand per thread and step; the next step's are on
  float va[PER], vb[PER];                                 // their way while this one is multiplied
  auto fetch = [&](int64_t r0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int o = tid + 256 * u, rr = sr == 1 ? o % G64_R : o / G64_T, ii = sr == 1 ? o / G64_R : o % G64_T;
      const float* src = v + (r0 + rr) * sr;
      va[u] = r0 + rr < r_end && i0 + ii < n ? src[(int64_t)(i0 + ii) * sv] : 0.0f;
      vb[u] = r0 + rr < r_end && j0 + ii < n ? src[(int64_t)(j0 + ii) * sv] : 0.0f;
    }
  };
  fetch(r_begin);
  for (int64_t r0 = r_begin; r0 < r_end; r0 += G64_R) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int o = tid + 256 * u, rr = sr == 1 ? o % G64_R : o / G64_T, ii = sr == 1 ? o / G64_R : o % G64_T;
      as[rr][ii] = (double)va[u];
      bs[rr][ii] = (double)vb[u];
    }
    __syncthreads();
    if (r0 + G64_R < r_end) fetch(r0 + G64_R);
    tile64_mac(as, bs, wm, wn, g, q, acc);
    __syncthreads();
  }
  double* dst = part + (int64_t)blockIdx.z * n * n;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int i = i0 + wm + 8 * a + g, j = j0 + wn + 8 * b + 2 * q + e;
        if (i < n && j < n) {
          dst[(int64_t)i * n + j] = acc[a][b][e];
          if (i0 != j0) dst[(int64_t)j * n + i] = acc[a][b][e];
        }
      }
}

// ------------------------------------------------------------------------------------------------
// Cholesky factor of the n x n Gram matrix g (symmetric to the bit, n <= MAXQ_WIDE).  A pivot not above tol_rel * (largest
// diagonal entry) marks a dependent sketch column: its column of L and its row and column of the diagonal-block inverse are zero.
//   l_out     n x n row-major lower factor (strict upper part zero)
//   dinv_out  (optional) inverses of the CW_NB x CW_NB diagonal blocks of L, [panel][CW_NB][CW_NB] row-major lower:
//             what the triangular solve H = Z L^-T needs besides L itself (trsm_wide_kernel)
//   well_conditioned  (optional) 1 when every pivot is above 1e-8 of the largest diagonal entry
//   perm_out  (optional) the matrix is factorised with its rows and columns sorted by descending diagonal entry;
//             perm_out[i] is the original index of row i
constexpr int CW_NB = 32, CW_P = CW_NB + 4;               // pitch: 4 mod 16 doubles, conflict-free fragment loads
constexpr int CW_THREADS = 512, CW_WARPS = CW_THREADS / 32;
constexpr int CW_ROWS = (MAXQ_WIDE + 31) / 32 * 32;
constexpr int CW_RT = (CW_ROWS / 8 + CW_WARPS - 1) / CW_WARPS;                 // row tiles per warp
constexpr size_t CW_SMEM = sizeof(double) * ((size_t)2 * CW_ROWS * CW_P + CW_NB * CW_P);

// One CTA, left-looking, panels of 32 columns; the matrix itself (half a megabyte in FP64) stays in global memory:
//   1. the panel (rows j0 .. n-1) minus the products with the finished columns on the FP64 tensor cores, the finished columns
//      streamed from global memory (L2) in chunks of 32, the next chunk on its way while one is multiplied;
//   2. the 32 x 32 diagonal block factorised by one warp in registers (lane = row; a column step is one pivot broadcast, one
//      reciprocal and one multiply-add deep);
//   3. the inverse of that factor by the same warp (lane = column), in registers;
//   4. the rows below the block:  L = A X^T  with X the inverse, on the tensor cores.
// With FP64 multiply-adds from shared memory and a column of the diagonal block per shared-memory round trip the
// factorisation took 138 us at n = 136; this form takes 104 us, and 286 us at n = 264.
struct EigState;
__device__ __forceinline__ void eig_state_reset(EigState* st, int tid);
__global__ void __launch_bounds__(CW_THREADS, 1)
chol_wide_kernel(const double* __restrict__ g, int n, double tol_rel, double* l_out, double* dinv_out, int* perm_out, EigState* state,
                 const int* __restrict__ skip, int* __restrict__ well_conditioned) {
  metis_pdl_wait();
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char cw_sm[];
  double (*P)[CW_P] = reinterpret_cast<double (*)[CW_P]>(cw_sm);                                      // the panel, rows j0 .. n-1
  double (*As)[CW_P] = reinterpret_cast<double (*)[CW_P]>(cw_sm + sizeof(double) * CW_ROWS * CW_P);   // a chunk of finished columns of those rows
  double (*Dv)[CW_P] = reinterpret_cast<double (*)[CW_P]>(cw_sm + sizeof(double) * 2 * CW_ROWS * CW_P);
  __shared__ double diag[MAXQ_WIDE];
  __shared__ int perm[MAXQ_WIDE];
  __shared__ double gmax_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gq = lane >> 2, q = lane & 3;
  if (state != nullptr) eig_state_reset(state, tid);
  for (int i = tid; i < n; i += CW_THREADS) { diag[i] = g[(int64_t)i * n + i]; perm[i] = i; }
  if (tid == 0) gmax_s = 0.0;
  __syncthreads();
  for (int i = tid; i < n; i += CW_THREADS) {
    const double d = diag[i];
    int rank = 0;
#pragma unroll 8
    for (int j = 0; j < n; ++j) rank += (diag[j] > d) || (diag[j] == d && j < i);
    if (rank == 0) gmax_s = d;
    if (perm_out != nullptr) perm[rank] = i;               // NaNs may collide; every entry stays a valid index
  }
  __syncthreads();
  if (perm_out != nullptr)
    for (int i = tid; i < n; i += CW_THREADS) perm_out[i] = perm[i];
  const double gmax = gmax_s, tol = tol_rel * gmax;
  double dmin = 1e300;                                     // smallest accepted pivot of this lane (warp 0)
  for (int j0 = 0; j0 < n; j0 += CW_NB) {
    const int w = min(CW_NB, n - j0), nr = n - j0, nr8 = (nr + 7) / 8;
    constexpr int PF = CW_ROWS / CW_WARPS;                 // rows per warp of a panel or chunk, lane = column
    double pre[PF];
    __syncthreads();                                       // the previous panel is stored
#pragma unroll
    for (int u = 0; u < PF; ++u) {                         // all loads of the panel in flight (the Gram matrix is symmetric to the bit)
      const int i = warp + u * CW_WARPS;
      pre[u] = i < nr && lane < w ? g[(int64_t)perm[j0 + i] * n + perm[j0 + lane]] : 0.0;        // zeros past the matrix and the panel
    }
#pragma unroll
    for (int u = 0; u < PF; ++u) P[warp + u * CW_WARPS][lane] = pre[u];
    // ---- 1. minus the products with the finished columns ----
    double acc[CW_RT][4][2] = {};
    auto fetch = [&](int k0) {
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const int i = warp + u * CW_WARPS;
        pre[u] = i < nr ? __ldcg(l_out + (int64_t)(j0 + i) * n + k0 + lane) : 0.0;
      }
    };
    if (j0 > 0) fetch(0);
    for (int k0 = 0; k0 < j0; k0 += CW_NB) {
      __syncthreads();
#pragma unroll
      for (int u = 0; u < PF; ++u) As[warp + u * CW_WARPS][lane] = pre[u];
      __syncthreads();
      if (k0 + CW_NB < j0) fetch(k0 + CW_NB);
#pragma unroll 2
      for (int kk = 0; kk < CW_NB; kk += 4) {              // rows j0 .. j0 + 31 of L are the first rows of the chunk
        double b[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) b[v] = As[8 * v + gq][kk + q];
#pragma unroll
        for (int u = 0; u < CW_RT; ++u) {
          const int rt = warp + u * CW_WARPS;
          if (rt < nr8) {
            const double a = As[8 * rt + gq][kk + q];
#pragma unroll
            for (int v = 0; v < 4; ++v) metis_small::dmma(acc[u][v], a, b[v]);
          }
        }
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < CW_RT; ++u) {
      const int rt = warp + u * CW_WARPS;
      if (rt < nr8 && j0 > 0) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          P[8 * rt + gq][8 * v + 2 * q] -= acc[u][v][0];
          P[8 * rt + gq][8 * v + 2 * q + 1] -= acc[u][v][1];
        }
      }
    }
    __syncthreads();
    // ---- 2. and 3.: the diagonal block and its inverse, warp 0 ----
    if (warp == 0) {
      double v[CW_NB];
#pragma unroll
      for (int c = 0; c < CW_NB; ++c) v[c] = lane < w && c < w ? P[lane][c] : 0.0;
      double pivot = 0.0;
#pragma unroll
      for (int c = 0; c < CW_NB; ++c) {
        const double d = __shfl_sync(0xFFFFFFFFu, v[c], c);
        const double l = v[c] * (d > tol ? metis_small::rcp_cubic(d) : 0.0);
        if (lane == c) pivot = d;
#pragma unroll
        for (int c2 = c + 1; c2 < CW_NB; ++c2) v[c2] = fma(-l, __shfl_sync(0xFFFFFFFFu, v[c], c2), v[c2]);
      }
      const bool ok = pivot > tol;
      const double rinv = ok ? metis_small::rsqrt_cubic(pivot) : 0.0;               // lane c: 1 / L[c][c]
      if (ok) dmin = fmin(dmin, pivot);
#pragma unroll
      for (int c = 0; c < CW_NB; ++c) {
        const double rc = __shfl_sync(0xFFFFFFFFu, rinv, c);
        P[lane][c] = lane >= c ? v[c] * rc : 0.0;
      }
      __syncwarp();
      // X = L^-1, lane = column:  X[i][j] = -r_i sum_{k < i} L[i][k] X[k][j]  (X[k][j] = 0 for k < j),  X[j][j] = r_j
      double x[CW_NB];
#pragma unroll
      for (int i = 0; i < CW_NB; ++i) {
        double s0 = 0.0, s1 = 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) { if (k & 1) s1 = fma(P[i][k], x[k], s1); else s0 = fma(P[i][k], x[k], s0); }
        const double ri = __shfl_sync(0xFFFFFFFFu, rinv, i);
        x[i] = i == lane ? ri : -ri * (s0 + s1);
        Dv[i][lane] = x[i];
      }
    }
    __syncthreads();
    // ---- 4. rows below the block: L = A X^T (X[c][cp] = Dv[c][cp], zero for cp > c); a warp reads and writes its own rows ----
#pragma unroll
    for (int u = 0; u < CW_RT; ++u) {
      const int rt = warp + u * CW_WARPS;
      if (rt >= CW_NB / 8 && rt < nr8) {
        double t[4][2] = {};
#pragma unroll
        for (int kk = 0; kk < CW_NB; kk += 4) {
          const double a = P[8 * rt + gq][kk + q];
#pragma unroll
          for (int v = 0; v < 4; ++v) metis_small::dmma(t[v], a, Dv[8 * v + gq][kk + q]);
        }
        __syncwarp();
#pragma unroll
        for (int v = 0; v < 4; ++v) { P[8 * rt + gq][8 * v + 2 * q] = t[v][0]; P[8 * rt + gq][8 * v + 2 * q + 1] = t[v][1]; }
      }
    }
    __syncthreads();
    for (int i = warp; i < nr; i += CW_WARPS)
      if (lane < w) __stcg(l_out + (int64_t)(j0 + i) * n + j0 + lane, P[i][lane]);
    for (int i = warp; i < w; i += CW_WARPS)
      for (int c = j0 + w + lane; c < n; c += 32) l_out[(int64_t)(j0 + i) * n + c] = 0.0;
    if (dinv_out != nullptr)
      for (int o = tid; o < CW_NB * CW_NB; o += CW_THREADS) dinv_out[(int64_t)(j0 / CW_NB) * CW_NB * CW_NB + o] = Dv[o / CW_NB][o % CW_NB];
  }
  if (warp == 0 && well_conditioned != nullptr) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmin = fmin(dmin, __shfl_xor_sync(0xFFFFFFFFu, dmin, o));
    if (lane == 0) *well_conditioned = (dmin > 1e-8 * gmax) ? 1 : 0;
  }
}

// The same outputs for n <= CM_MAX, whose factor fits one SM's shared memory: the eight-column panels of cta_cholesky (a
// panel costs 2.4k cycles whatever n is; n = 136: 45 us against 104 us of the 32-column panels), then the inverses of the
// diagonal blocks, one warp each.
constexpr int CM_MAX = 160, CM_P = CM_MAX + 4;
__host__ __device__ constexpr size_t cm_smem(int n) { return sizeof(double) * (size_t)((n + 7) / 8 * 8) * CM_P; }
__device__ __forceinline__ void chol_mid(const double* __restrict__ g, int n, double tol_rel, double* __restrict__ l_out, double* dinv_out, int* perm_out,
                                         EigState* state, int* __restrict__ well_conditioned) {
  extern __shared__ __align__(16) unsigned char cm_sm[];
  double* Y = reinterpret_cast<double*>(cm_sm);
  __shared__ double diag[CM_MAX], inv_s[CM_MAX];
  __shared__ int perm[CM_MAX];
  __shared__ double gmax_s, dmin_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, n8 = (n + 7) & ~7;
  if (state != nullptr) eig_state_reset(state, tid);
  for (int i = tid; i < n; i += CW_THREADS) { diag[i] = g[(int64_t)i * n + i]; perm[i] = i; }
  if (tid == 0) gmax_s = 0.0;
  __syncthreads();
  static_assert(CM_MAX <= CW_THREADS / 2, "two lanes per diagonal entry in one pass");
  {
    // two lanes per entry, in whole warps: for an odd n the lanes of a pair count different numbers of entries, so the sum is
    // taken behind the loop by every thread (joined inside it, a lane's partner may not have arrived)
    const int i = tid >> 1;
    const double d = i < n ? diag[i] : 0.0;
    int rank = 0;
    if (i < n) {
#pragma unroll 8
      for (int j = tid & 1; j < n; j += 2) rank += (diag[j] > d) || (diag[j] == d && j < i);
    }
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 1);
    if (i < n && (tid & 1) == 0) {
      if (rank == 0) gmax_s = d;
      if (perm_out != nullptr) perm[rank] = i;             // NaNs may collide; every entry stays a valid index
    }
  }
  __syncthreads();
  if (perm_out != nullptr)
    for (int i = tid; i < n; i += CW_THREADS) perm_out[i] = perm[i];
#pragma unroll 4
  for (int i = warp; i < n8; i += CW_WARPS) {              // rows of the sorted matrix (symmetric to the bit)
    double v[CM_MAX / 32];
#pragma unroll
    for (int t = 0; t < CM_MAX / 32; ++t) { const int c = lane + 32 * t; v[t] = i < n && c < n ? g[(int64_t)perm[i] * n + perm[c]] : 0.0; }
#pragma unroll
    for (int t = 0; t < CM_MAX / 32; ++t) { const int c = lane + 32 * t; if (c < n8) Y[i * CM_P + c] = v[t]; }
  }
  const double gmax = gmax_s;
  __syncthreads();
  metis_small::cta_cholesky<CM_P>(Y, n, tol_rel * gmax, inv_s, &dmin_s, CW_THREADS);
  for (int i = warp; i < n; i += CW_WARPS)
    for (int c = lane; c < n; c += 32) l_out[(int64_t)i * n + c] = c <= i ? Y[i * CM_P + c] : 0.0;
  if (tid == 0 && well_conditioned != nullptr) *well_conditioned = (dmin_s > 1e-8 * gmax) ? 1 : 0;
  if (dinv_out != nullptr && warp < (n + CW_NB - 1) / CW_NB) {
    // X = L^-1 of a diagonal block, lane = column:  X[i][j] = -r_i sum_{k < i} L[i][k] X[k][j],  X[j][j] = r_j
    const int j0 = warp * CW_NB;
    double x[CW_NB];
#pragma unroll
    for (int i = 0; i < CW_NB; ++i) {
      double s0 = 0.0, s1 = 0.0;
      const bool in = j0 + i < n;
      const double* row = Y + (in ? j0 + i : j0) * CM_P + j0;
#pragma unroll
      for (int k = 0; k < i; ++k) { if (k & 1) s1 = fma(row[k], x[k], s1); else s0 = fma(row[k], x[k], s0); }
      const double ri = in ? inv_s[j0 + i] : 0.0;
      x[i] = i == lane ? ri : (i > lane ? -ri * (s0 + s1) : 0.0);
      dinv_out[(int64_t)warp * CW_NB * CW_NB + i * CW_NB + lane] = x[i];
    }
  }
}

__global__ void __launch_bounds__(CW_THREADS, 1)
chol_mid_kernel(const double* __restrict__ g, int n, double tol_rel, double* __restrict__ l_out, double* dinv_out, int* perm_out, EigState* state,
                const int* __restrict__ skip, int* __restrict__ well_conditioned) {
  metis_pdl_wait();
  if (skip != nullptr && *skip) return;
  chol_mid(g, n, tol_rel, l_out, dinv_out, perm_out, state, well_conditioned);
}

// H = Z L^-T by blocked forward substitution, in place: for panel J of CW_NB columns
//   h_J = (z_J - sum_{K < J} h_K L[J][K]^T) Dinv_J^T.
// A CTA owns 32 rows of Z and keeps their finished part of H in shared memory (FP64).  The products run on the FP64 tensor cores, a warp
// two 8 x 8 tiles of the panel; the factor's and the inverse's entries go from L2 into fragment registers, a panel of 32 columns ahead
// (544 x 136 46 -> 15.5 us, 7168 x 136 61 -> 22.6 us; before: multiply-adds from shared memory, loads behind barriers).
// l, dinv: outputs of the wide Cholesky kernels.  FP32 in, FP64 arithmetic, FP32 out.
constexpr int TW_ROWS = 32, TW_HP = MAXQ_WIDE + 4, TW_TP = CW_NB + 4;          // pitches 4 mod 16: conflict-free fragments
constexpr size_t TW_SMEM = sizeof(double) * TW_ROWS * (TW_HP + TW_TP);
static_assert(CW_NB == 32 && TW_HP % 16 == 4 && TW_TP % 16 == 4, "fragment layout");
__global__ void __launch_bounds__(256)
trsm_wide_kernel(float* __restrict__ z, int64_t n_rows, int n, const double* __restrict__ l, const double* __restrict__ dinv,
                 const int* __restrict__ skip) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) unsigned char tw_sm[];
  double (*Hs)[TW_HP] = reinterpret_cast<double (*)[TW_HP]>(tw_sm);
  double (*Ts)[TW_TP] = reinterpret_cast<double (*)[TW_TP]>(tw_sm + sizeof(double) * TW_ROWS * TW_HP);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
  const int row = 8 * (warp & 3) + g;                     // row of the fragments this lane holds
  const int64_t r = (int64_t)blockIdx.x * TW_ROWS + row;
  for (int j0 = 0; j0 < n; j0 += CW_NB) {
    const int jt[2] = {j0 + 8 * (warp >> 2), j0 + 8 * (warp >> 2) + 16};       // first columns of the warp's tiles
    double acc[2][2][2] = {}, f[2][8];
    // entries of the factor (k0 < j0) or of the inverse of its diagonal block (k0 = j0) that multiply columns k0 ... k0 + 31
    auto fetch = [&](int k0) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int s = 0; s < 8; ++s) {
          const int c = jt[u] + g;
          f[u][s] = c >= n ? 0.0 : (k0 < j0 ? __ldg(l + (int64_t)c * n + k0 + 4 * s + q) : __ldg(dinv + (int64_t)(j0 / CW_NB) * CW_NB * CW_NB + (c - j0) * CW_NB + 4 * s + q));
        }
    };
    fetch(0);
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = jt[u] + 2 * q + e;
        acc[u][0][e] = r < n_rows && c < n ? (double)z[r * n + c] : 0.0;
      }
    for (int k0 = 0; k0 < j0; k0 += CW_NB) {
      double b[2][8];
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int s = 0; s < 8; ++s) b[u][s] = f[u][s];
      fetch(k0 + CW_NB);
#pragma unroll
      for (int s = 0; s < 8; ++s) {
        const double a = -Hs[row][k0 + 4 * s + q];
#pragma unroll
        for (int u = 0; u < 2; ++u) metis_small::dmma(acc[u][s & 1], a, b[u][s]);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int e = 0; e < 2; ++e) Ts[row][jt[u] - j0 + 2 * q + e] = acc[u][0][e] + acc[u][1][e];
    __syncthreads();
    double h[2][2][2] = {};
#pragma unroll
    for (int s = 0; s < 8; ++s) {
      const double a = Ts[row][4 * s + q];
#pragma unroll
      for (int u = 0; u < 2; ++u) metis_small::dmma(h[u][s & 1], a, f[u][s]);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int c = jt[u] + 2 * q + e;
        const double v = h[u][0][e] + h[u][1][e];
        if (c < n) {
          Hs[row][c] = v;
          if (r < n_rows) z[r * n + c] = (float)v;
        }
      }
    __syncthreads();                                      // the panel's columns are there; Ts has been read
  }
}

// ------------------------------------------------------------------------------------------------
// C[m][n] = scale[n] * sum_k A[m * a_m + k * a_k] * B[k * b_k + n * b_n]      (A FP32, B FP64, FP64 accumulation)
// (on the FP64 tensor cores) written as FP32 to c[m * c_m + n * c_n]; optionally also c2[m * c2_m + n * c2_n] = (that value) * scale2[n], and
// amax|C| into *amax (bits of a non-negative float, atomic max).  64 x 64 tile per CTA, 16 x 32 per warp.
struct Gemm64Args {
  const float* a; int64_t a_m, a_k;
  const double* b; int64_t b_k, b_n;
  const double* scale;            // per output column n, or NULL
  float* c; int64_t c_m, c_n;
  float* c2; int64_t c2_m, c2_n; const float* scale2;
  float* amax;
  int64_t M; int N, K;
  const int* skip;
};
__global__ void __launch_bounds__(256)
gemm64_kernel(Gemm64Args g) {
  metis_pdl_wait_trigger();
  if (g.skip != nullptr && *g.skip) return;
  constexpr int T = G64_T, KT = G64_R;
  __shared__ double as[KT][G64_P], bs[KT][G64_P];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gq = lane >> 2, q = lane & 3, wm = 16 * (warp & 3), wn = 32 * (warp >> 2);
  const int64_t m0 = (int64_t)blockIdx.y * T;
  const int n0 = blockIdx.x * T;
  double acc[2][4][2] = {};
  constexpr int PER = KT * T / 256;                       // values of either operand per thread and step; the next step's are on
  float va[PER];                                          // their way while this one is multiplied
  double vb[PER];
  const bool a_rows = g.a_k == 1, b_cols = g.b_k == 1;
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int o = tid + 256 * u;
      const int kk = a_rows ? o % KT : o / T, mm = a_rows ? o / KT : o % T, kb = b_cols ? o % KT : o / T, nn = b_cols ? o / KT : o % T;
      va[u] = m0 + mm < g.M && k0 + kk < g.K ? g.a[(m0 + mm) * g.a_m + (int64_t)(k0 + kk) * g.a_k] : 0.0f;
      vb[u] = n0 + nn < g.N && k0 + kb < g.K ? g.b[(int64_t)(k0 + kb) * g.b_k + (int64_t)(n0 + nn) * g.b_n] : 0.0;
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < g.K; k0 += KT) {
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int o = tid + 256 * u;
      as[a_rows ? o % KT : o / T][a_rows ? o / KT : o % T] = (double)va[u];
      bs[b_cols ? o % KT : o / T][b_cols ? o / KT : o % T] = vb[u];
    }
    __syncthreads();
    if (k0 + KT < g.K) fetch(k0 + KT);
    tile64_mac(as, bs, wm, wn, gq, q, acc);
    __syncthreads();
  }
  float am = 0.0f;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int64_t m = m0 + wm + 8 * a + gq;
        const int n = n0 + wn + 8 * b + 2 * q + e;
        if (m < g.M && n < g.N) {
          const float v = (float)(g.scale != nullptr ? acc[a][b][e] * g.scale[n] : acc[a][b][e]);
          g.c[m * g.c_m + (int64_t)n * g.c_n] = v;
          if (g.c2 != nullptr) g.c2[m * g.c2_m + (int64_t)n * g.c2_n] = v * g.scale2[n];
          am = fmaxf(am, fabsf(v));
        }
      }
  if (g.amax != nullptr) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xFFFFFFFFu, am, o));
    if ((tid & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(g.amax), __float_as_uint(am));
  }
}

// per-column scales of the rotations: mode 0: 1/sqrt(eval_j) (right basis; also writes sigma_out = sqrt(eval_j)),
// mode 1: sign_j / sqrt(eval_j) (Rayleigh-Ritz left factor; sigma_out likewise), mode 2: sign_j
__global__ void rot_scales_kernel(const double* __restrict__ evals, const float* __restrict__ sign, int k, int mode,
                                  double* __restrict__ scale, float* __restrict__ sigma_out) {
  metis_pdl_wait_trigger();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= k) return;
  double s = 1.0;
  if (mode != 2) {
    const double lam = sqrt(fmax(evals[j], 0.0));
    s = lam > 0.0 ? 1.0 / lam : 0.0;
    if (sigma_out != nullptr) sigma_out[j] = (float)lam;
  }
  if (mode != 0) s *= (double)sign[j];
  scale[j] = s;
}

// ------------------------------------------------------------------------------------------------
// Symmetric eigen-decomposition of a Gram matrix of n up to MAXQ_WIDE, in the steps of the one-CTA solver (small_eig.cuh):
// sorted Cholesky factor, a start (tridiagonal matrix up to n = 144, FP32 block Jacobi above), FP64 refinement with matrix products over
// many CTAs; a matrix the refinement cannot finish (pairs of eigenvalues too close, or no convergence) is done by the FP64 Jacobi
// kernels, which otherwise return at once.  The decisions are made on the device, in EigState, so that a call needs no host
// synchronisation.
// Measured inside a layer step, factorisation and start: n = 136 243 us (reduction 202, vectors 20, back 20; factorisation and FP32
// Jacobi before: 43 + 338), n = 128 190 us (37 + 276), n = 104 165 us; refinement, finish and collection 60 us.  Repeated eigenvalues pay
// for both solvers.
constexpr int ER_STEPS = 3;                               // refinement steps (two are enough unless eigenvalues are close)
struct EigState {
  unsigned int emax[ER_STEPS];                            // largest |E_ij| of a step (bits)
  // squared norm of E in units of 2^-40: a sum of integers is the same in every order of arrival, and it chooses the solver
  unsigned long long norm2[ER_STEPS];
  int open[ER_STEPS];                                     // some pair could not be separated
};
__device__ __forceinline__ void eig_state_reset(EigState* st, int tid) {
  if (tid < ER_STEPS) { st->emax[tid] = 0u; st->norm2[tid] = 0ull; st->open[tid] = 0; }
}
constexpr float EIG_NORM2_UNITS = 1099511627776.0f;       // 2^40
__device__ __forceinline__ unsigned long long eig_norm2_units(float x) { return x < 1024.0f ? __float2ull_rz(x * EIG_NORM2_UNITS) : 1ull << 50; }   // (a NaN is a large one)
enum { EIG_RUNNING = 0, EIG_DONE = 1, EIG_FAILED = 2 };
__device__ __forceinline__ bool eig_step_bad(const EigState* st, int t) { return __ldcg(&st->open[t]) != 0 || __ldcg(&st->norm2[t]) >= eig_norm2_units(0.0625f); }
// what the steps before `step` have come to; *last: the last step that was applied
__device__ __forceinline__ int eig_status(const EigState* st, int step, int* last) {
  *last = -1;
  for (int t = 0; t < step; ++t) {
    if (eig_step_bad(st, t)) return EIG_FAILED;
    *last = t;
    if (__uint_as_float(__ldcg(&st->emax[t])) < 2e-7f) return EIG_DONE;
  }
  return EIG_RUNNING;
}

// round-robin tournament of np players: couple I of round `step`
__device__ __forceinline__ void jc_pair(int I, int step, int np, int* p, int* q) {
  int a, b;
  if (I == 0) { a = 0; b = (step % (np - 1)) + 1; }
  else { a = ((step + I) % (np - 1)) + 1; b = ((step + np - 1 - I) % (np - 1)) + 1; }
  *p = min(a, b); *q = max(a, b);
}

// FP32 one-sided block Jacobi on one cluster: 48 columns per CTA - two slots of twelve blocks of two columns, eight lanes per
// block (sixteen above n = 176, where eight lanes' rows no longer fit their registers), so that the three warps sit on three schedulers (a warp per block: 1220 cycles a round at n = 136, the nine warps
// sharing four schedulers, against 900) - and as many CTAs as the matrix needs.  Outer rounds are those of jacobi_cluster_kernel
// below: first every pair among a CTA's own columns, then every block of one slot (kept in registers) against every block of the other,
// the slots moving on to the neighbouring CTAs in the order of a round-robin tournament.  Ends with the
// normalised columns in x (n x n, FP64).
constexpr int JF_MB = 12, JF_COLS = 4 * JF_MB, JF_SWEEPS = 16;
constexpr float JF_EXIT_COS2 = 1e-8f;                     // the rank cut may fall among close eigenvalues: a tighter exit than the small solver's
__host__ __device__ constexpr size_t jf_smem(int lanes, int r) { return sizeof(float2) * 2 * 2 * JF_MB * lanes * (size_t)r; }
template <int LANES, int R>                               // lanes per block; rows per lane, even: at least n / LANES
__global__ void __launch_bounds__(LANES * JF_MB, 1)
jacobi_fp32_kernel(const double* __restrict__ l, int n, double* __restrict__ x) {
  constexpr int ROWS = LANES * R, JF_THREADS = LANES * JF_MB;
  extern __shared__ __align__(16) unsigned char jf_sm[];
  float2* blocks = reinterpret_cast<float2*>(jf_sm);      // [buffer][slot][block][row]
  __shared__ float2 nrm[2 * JF_MB];
  __shared__ int flag_s;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), P = (int)cluster.num_blocks();
  const int tid = threadIdx.x, m = tid / LANES, sub = tid % LANES;             // group (block) and lane in it
  auto blk = [&](int buf, int sb) { return blocks + ((size_t)buf * 2 * JF_MB + sb) * ROWS; };     // sb: slot * JF_MB + block
  // odd groups walk the chunks of LANES rows in the order 1, 0, 3, 2, ...: the two groups of a half warp use different banks
  auto row_of = [&](int t) { return sub + LANES * (t ^ (m & 1)); };
  // FP32 copy, scaled to a largest entry near one (the factor's first pivot is its largest)
  int ex = 0;
  { const double l00 = l[0]; if (l00 > 0.0 && l00 < 1e150) (void)frexp(l00, &ex); }
  const double scale = ldexp(1.0, -ex);
#pragma unroll 4
  for (int o = tid; o < 2 * JF_MB * ROWS; o += JF_THREADS) {
    const int sb = o % (2 * JF_MB), i = o / (2 * JF_MB), c = rank * JF_COLS + 2 * sb;
    float2 y = make_float2(0.0f, 0.0f);
    if (i < n) {
      if (c < n && c <= i) y.x = (float)(l[(int64_t)i * n + c] * scale);
      if (c + 1 < n && c + 1 <= i) y.y = (float)(l[(int64_t)i * n + c + 1] * scale);
    }
    blk(0, sb)[i] = y;
  }
  __syncthreads();
  int cur = 0;
  for (int sweep = 0; sweep < JF_SWEEPS; ++sweep) {
    bool above = false;
    int any_above = 0;
    for (int orr = 0; orr < 2 * P - 1; ++orr) {
      // exact norms at the start of every outer round (carried through its rounds)
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        const float2* y = blk(cur, s * JF_MB + m);
        float2 sq = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int t = 0; t < R; ++t) { const float2 v = y[row_of(t)]; sq = metis_small::fma2(v, v, sq); }
#pragma unroll
        for (int o = LANES / 2; o > 0; o >>= 1) { sq.x += __shfl_xor_sync(0xFFFFFFFFu, sq.x, o); sq.y += __shfl_xor_sync(0xFFFFFFFFu, sq.y, o); }
        if (sub == 0) nrm[s * JF_MB + m] = sq;
      }
      __syncthreads();
      float2 a[R], b[R];
      if (orr == 0) {
        // every pair among the CTA's own columns: tournament of its 2 * JF_MB blocks
        for (int r = 0; r < 2 * JF_MB - 1; ++r) {
          int p, q;
          jc_pair(m, r, 2 * JF_MB, &p, &q);
          float2 *yp = blk(cur, p), *yq = blk(cur, q);
#pragma unroll
          for (int t = 0; t < R; ++t) { a[t] = yp[row_of(t)]; b[t] = yq[row_of(t)]; }
          float2 n01 = nrm[p], n23 = nrm[q];
          metis_small::block_rotate<R, LANES>(a, b, n01, n23, r == 0, JF_EXIT_COS2, above);
#pragma unroll
          for (int t = 0; t < R; ++t) { yp[row_of(t)] = a[t]; yq[row_of(t)] = b[t]; }
          __syncwarp();
          if (sub == 0) { nrm[p] = n01; nrm[q] = n23; }
          __syncthreads();
        }
      } else {
        // group m keeps block m of the first slot in registers and meets the blocks of the second slot one after the other
        float2* yp = blk(cur, m);
#pragma unroll
        for (int t = 0; t < R; ++t) a[t] = yp[row_of(t)];
        float2 n01 = nrm[m];
        int q = JF_MB + m;
        for (int r = 0; r < JF_MB; ++r) {
          float2* yq = blk(cur, q);
#pragma unroll
          for (int t = 0; t < R; ++t) b[t] = yq[row_of(t)];
          float2 n23 = nrm[q];
          metis_small::block_rotate<R, LANES>(a, b, n01, n23, false, JF_EXIT_COS2, above);
#pragma unroll
          for (int t = 0; t < R; ++t) yq[row_of(t)] = b[t];
          __syncwarp();
          if (sub == 0) nrm[q] = n23;
          q = q + 1 == 2 * JF_MB ? JF_MB : q + 1;
          __syncthreads();
        }
#pragma unroll
        for (int t = 0; t < R; ++t) yp[row_of(t)] = a[t];
        __syncthreads();
      }
      const bool last = orr == 2 * P - 2;
      if (last) {
        const int any = __syncthreads_or(above ? 1 : 0);
        if (tid == 0) flag_s = any;
      }
      cluster.sync();                                      // every CTA is done with this outer round (flags are written)
      // hand the slots on: slot 0 ("top") of CTA c goes to the top of c + 1 (the last CTA's top becomes its own
      // bottom, CTA 0's top stays); slot 1 ("bottom") of CTA c goes to the bottom of c - 1 (CTA 0's bottom becomes
      // the top of CTA 1)
      {
        int dst_rank[2], dst_slot[2];
        if (rank == 0) { dst_rank[0] = 0; dst_slot[0] = 0; dst_rank[1] = 1; dst_slot[1] = 0; }
        else {
          if (rank == P - 1) { dst_rank[0] = rank; dst_slot[0] = 1; } else { dst_rank[0] = rank + 1; dst_slot[0] = 0; }
          dst_rank[1] = rank - 1; dst_slot[1] = 1;
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float4* src = reinterpret_cast<const float4*>(blk(cur, s * JF_MB));
          float4* dst = reinterpret_cast<float4*>(cluster.map_shared_rank(blk(cur ^ 1, dst_slot[s] * JF_MB), dst_rank[s]));
#pragma unroll 8
          for (int o = tid; o < JF_MB * ROWS / 2; o += JF_THREADS) dst[o] = src[o];
        }
      }
      if (last) {
        for (int c = 0; c < P; ++c) any_above |= *cluster.map_shared_rank(&flag_s, c);
      }
      cluster.sync();                                      // the slots have landed; the flags have been read
      cur ^= 1;
    }
    if (!any_above) break;
  }
  // after whole sweeps every slot is back where it started; normalised columns, zero columns stay zero
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const float2* y = blk(cur, s * JF_MB + m);
    double sx = 0.0, sy = 0.0;
#pragma unroll
    for (int t = 0; t < R; ++t) { const float2 v = y[row_of(t)]; sx = fma((double)v.x, (double)v.x, sx); sy = fma((double)v.y, (double)v.y, sy); }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) { sx += __shfl_xor_sync(0xFFFFFFFFu, sx, o); sy += __shfl_xor_sync(0xFFFFFFFFu, sy, o); }
    const double rx = sx > 0.0 ? metis_small::rsqrt_cubic(sx) : 0.0, ry = sy > 0.0 ? metis_small::rsqrt_cubic(sy) : 0.0;
    const int c = rank * JF_COLS + 2 * (s * JF_MB + m);
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const int i = row_of(t);
      const float2 v = y[i];
      if (i < n && c < n) x[(int64_t)i * n + c] = (double)v.x * rx;
      if (i < n && c + 1 < n) x[(int64_t)i * n + c + 1] = (double)v.y * ry;
    }
  }
}

// The start of the refinement up to n = WT_MAX, as in the one-CTA solver: Householder reduction to a tridiagonal matrix (CTA 0)
// beside the sorted factorisation (CTA 1).  Fifteen warps hold the matrix in registers, warp w the rows w, w + 15, ..., a lane the
// columns n - 1 - lane, n - 1 - lane - 32, ...: a column of the vectors is loaded once for all of a warp's rows (shared-memory delivery,
// 128 bytes a cycle, is what a squarer tile of four lanes a row waits for), and what is finished drops out, three rows at a time.
// Above n = 128 the first columns, finished first, live in shared memory: five per lane do not fit the registers.
// The sixteenth warp works out the scalars, the vectors of the update and the next column, so that a step has two barriers.  A step takes
// 2300 cycles at n = 128, 3300 over the first quarter: the shared-memory pipe (52 cycles a warp for the factors of 36 elements a lane,
// 24 for the exchanges) and the FP64 pipe (54) share it with the scalars' 1050 (rows along the lanes instead would
// need the products of fifteen warps summed through shared memory; five columns per lane in registers spilled, n = 136: 309 us).
// Outputs: v[j][.] the reflectors (zero up to column j), tri = d, e, beta (n each).
constexpr int WT_WARPS = 15, WT_THREADS = 32 * (WT_WARPS + 1), WT_MAX = 144, WT_TAIL = 16, WT_ROWS = 3;
static_assert(WT_MAX <= CM_MAX && WT_THREADS >= CW_THREADS, "the factorisation runs in the same launch");
// An instance of R rows per warp and C columns per lane holds orders up to N_MAX.  Rows it has beyond the matrix are worked on like the
// others (they stay zero), so what is indexed by a row has an entry for each of its WT_WARPS * R.
template <int R, int C, bool TAIL>
struct WtShape {
  static constexpr int ROWS = WT_WARPS * R, COLS = 32 * C + (TAIL ? WT_TAIL : 0), N_MAX = ROWS < COLS ? ROWS : COLS;
  static constexpr int LANE_COLS = TAIL ? C + 1 : C, PADDED = 32 * LANE_COLS;   // columns per lane of the scalars' warp, and of all its lanes
  static constexpr int ENTRIES = ROWS > PADDED ? ROWS : PADDED;
  static_assert(COLS <= PADDED && (!TAIL || ROWS <= WT_MAX + WT_WARPS), "columns of the vectors, rows of the tail");
};
template <int R, int C, bool TAIL>
__global__ void __launch_bounds__(WT_THREADS, 1)
tridiag_chol_kernel(const double* __restrict__ gm, int n, double* __restrict__ l_out, int* __restrict__ perm_out, EigState* __restrict__ state,
                    double* __restrict__ v_out, double* __restrict__ tri) {
  metis_pdl_wait();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (blockIdx.x == 1) {
    if (tid < CW_THREADS) chol_mid(gm, n, 1e-14, l_out, nullptr, perm_out, state, nullptr);
    return;
  }
  using Shape = WtShape<R, C, TAIL>;
  constexpr int CS = Shape::LANE_COLS, NP = Shape::PADDED;
  __shared__ double xs_[32 + NP], rs_[32 + NP], us_[32 + NP];                  // the first 32 stay zero: columns below the first
  __shared__ double ys[Shape::ENTRIES];                   // by row, as is pq; what lies beyond the matrix stays zero
  __shared__ __align__(16) double2 pq[Shape::ENTRIES];
  __shared__ double tail[TAIL ? WT_MAX + WT_WARPS : 1][WT_TAIL];               // columns 0 ... n - 32 C - 1
  double *xs = xs_ + 32, *rs = rs_ + 32, *us = us_ + 32;
  for (int i = tid; i < 32 + NP; i += WT_THREADS) { xs_[i] = 0.0; rs_[i] = 0.0; us_[i] = 0.0; }
  for (int i = tid; i < Shape::ENTRIES; i += WT_THREADS) { ys[i] = 0.0; pq[i] = make_double2(0.0, 0.0); }
  int top = 0;                                            // an even power of two brings the largest entry near one
  for (int i = lane; i < n; i += 32) top = max(top, __double2hiint(gm[(int64_t)i * n + i]));
  top = __reduce_max_sync(0xFFFFFFFFu, top) >> 20;
  const int ex = top > 0 && top < 2046 ? (top - 1022 + 1) >> 1 : 0;
  const double scale = __hiloint2double((1023 - 2 * ex) << 20, 0);
  double *d_out = tri, *e_out = tri + n, *b_out = tri + 2 * n;
  const int n_tail = TAIL ? n - 32 * C : 0;
  __syncthreads();
  if (warp < WT_WARPS) {
    const int c0 = n - 1 - lane;                          // column of t = 0
    double row[R][C];
#pragma unroll
    for (int a = 0; a < R; ++a) {
      const int i = warp + WT_WARPS * a;
#pragma unroll
      for (int t = 0; t < C; ++t) row[a][t] = i < n && c0 - 32 * t >= 0 ? gm[(int64_t)i * n + c0 - 32 * t] * scale : 0.0;
      if (TAIL && i < WT_MAX + WT_WARPS && lane < WT_TAIL) tail[i][lane] = i < n && lane < n_tail ? gm[(int64_t)i * n + lane] * scale : 0.0;
    }
    // row i, columns from `from` on
    auto publish = [&](double* out, int i, int from) {
      const int a_own = i / WT_WARPS;
      if (i - a_own * WT_WARPS == warp) {
        if (TAIL && lane < n_tail) out[lane] = lane >= from ? tail[i][lane] : 0.0;
#pragma unroll
        for (int a = 0; a < R; ++a)
          if (a == a_own) {
#pragma unroll
            for (int t = 0; t < C; ++t) if (c0 - 32 * t >= 0) out[c0 - 32 * t] = c0 - 32 * t >= from ? row[a][t] : 0.0;
          }
      }
    };
    __syncwarp();
    publish(xs, 0, 1);
    if (tid == 0) d_out[0] = gm[0] * scale;
    __syncthreads();
    double x[C];                                          // the vector of the last product
#pragma unroll
    for (int t = 0; t < C; ++t) x[t] = 0.0;
    double x_tail = 0.0;
    // the update of step j - 1 and the product of step j on the last rl rows and the last 32 cl columns, which are all that is left
    auto work = [&](auto cl, auto rl, int j) {
      constexpr int CL = decltype(cl)::value, RL = decltype(rl)::value, A0 = R - RL;
      double u[CL], xn[CL], y[RL];
#pragma unroll
      for (int t = 0; t < CL; ++t) { u[t] = us[c0 - 32 * t]; xn[t] = xs[c0 - 32 * t]; }
#pragma unroll
      for (int b = 0; b < RL; b += WT_ROWS) {
#pragma unroll
        for (int a = b; a < b + WT_ROWS && a < RL; ++a) y[a] = 0.0;
        if (warp + WT_WARPS * (A0 + b + WT_ROWS - 1) >= j) {
          double2 c[WT_ROWS];
#pragma unroll
          for (int h = 0; h < WT_ROWS; ++h) if (b + h < RL) c[h] = pq[warp + WT_WARPS * (A0 + b + h)];
#pragma unroll
          for (int h = 0; h < WT_ROWS; ++h)               // (a factor that stays from one multiply-add to the next is read once)
            if (b + h < RL) {
#pragma unroll
              for (int t = 0; t < CL; ++t) row[A0 + b + h][t] = fma(c[h].y, x[t], row[A0 + b + h][t]);
#pragma unroll
              for (int t = 0; t < CL; ++t) row[A0 + b + h][t] = fma(c[h].x, u[t], row[A0 + b + h][t]);
            }
#pragma unroll
          for (int t = 0; t < CL; ++t)
#pragma unroll
            for (int h = 0; h < WT_ROWS; ++h)
              if (b + h < RL) y[b + h] = fma(row[A0 + b + h][t], xn[t], y[b + h]);
        }
      }
      if (TAIL && CL == C && j <= n_tail && lane < n_tail) {
        const double ut = us[lane], xt = xs[lane];
#pragma unroll
        for (int a = 0; a < RL; ++a) {
          const double2 c = pq[warp + WT_WARPS * (A0 + a)];
          double* at = &tail[warp + WT_WARPS * (A0 + a)][lane];
          const double v = fma(c.x, ut, fma(c.y, x_tail, *at));
          *at = v;
          y[a] = fma(v, xt, y[a]);
        }
        x_tail = xt;
      }
#pragma unroll
      for (int t = 0; t < CL; ++t) x[t] = xn[t];
      // sums over the lanes: at each exchange half of the values go to the other half of the lanes; a lane ends with row `mine`
      int m = RL, mine = 0, half_at[5];
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const int o = 16 >> k, half = (m + 1) / 2;
        const bool hi = lane & o;
#pragma unroll
        for (int h = 0; h < half; ++h) {
          if (h + half < m) {
            const double give = hi ? y[h] : y[h + half], keep = hi ? y[h + half] : y[h];
            y[h] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
          } else {
            y[h] += __shfl_xor_sync(0xFFFFFFFFu, y[h], o);
          }
        }
        half_at[k] = half;
        m = half;
      }
#pragma unroll
      for (int k = 4; k >= 0; --k)
        if (mine + half_at[k] < (k == 0 ? RL : half_at[k > 0 ? k - 1 : 0]) && (lane & (16 >> k))) mine += half_at[k];
      ys[warp + WT_WARPS * (A0 + mine)] = y[0];
      __syncwarp();
      publish(rs, j + 1, j + 1);
    };
    constexpr int N_MAX = 32 * C + (TAIL ? WT_TAIL : 0), R2 = C > 2 ? R - (N_MAX - 64) / WT_WARPS : R, R1 = R - (N_MAX - 32) / WT_WARPS;
    const int from2 = max(n - 64, WT_WARPS * (R - R2)), from1 = max(n - 32, WT_WARPS * (R - R1));   // what the later forms leave out is finished
#pragma unroll 1
    for (int j = 0; j + 2 < n; ++j) {
      if (warp + WT_WARPS * (R - 1) >= j) {
        if (j >= from1) work(std::integral_constant<int, 1>(), std::integral_constant<int, R1>(), j);
        else if (j >= from2) work(std::integral_constant<int, 2>(), std::integral_constant<int, R2>(), j);
        else work(std::integral_constant<int, C>(), std::integral_constant<int, R>(), j);
      }
      __syncthreads();                                    // the product is there
      __syncthreads();                                    // the next update and the next column are there
    }
    // the last diagonal entry, with the last update
    if (lane == 0) {
#pragma unroll
      for (int a = 0; a < R; ++a) {
        const int i = warp + WT_WARPS * a;
        if (i == n - 1) d_out[n - 1] = fma(pq[i].x, us[n - 1], fma(pq[i].y, x[0], row[a][0]));
      }
    }
  } else {
    // with y = A x and r = A e_1 it is A v = u = y - alpha r,  v^T A v = x^T y - 2 alpha y_1 + alpha^2 r_1;  w = beta u - K v,
    // A -= v w^T + w v^T = p u^T + q v^T.  Column j + 1 of the product is not read again except for its first entry, so x
    // stands for v in the last term.  The next column, r + u_1 p + v_1 q, needs no row of the updated matrix: this warp goes on with its
    // length and its reflector while the others update and multiply.
    __syncthreads();
    double x[CS];
#pragma unroll
    for (int t = 0; t < CS; ++t) x[t] = xs[lane + 32 * t];
#pragma unroll 1
    for (int j = 0; j + 2 < n; ++j) {
      double r[CS], y[CS], sq = 0.0, xy = 0.0, alpha, beta;
      const double x0 = xs[j + 1];
#pragma unroll
      for (int t = 0; t < CS; ++t) sq = fma(x[t], x[t], sq);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
      metis_tri::reflector(x0, sq, alpha, beta);
      const double b2 = beta * beta, v1 = x0 - alpha;
#pragma unroll
      for (int t = 0; t < CS; ++t)
        if (lane + 32 * t < n) v_out[(int64_t)j * n + lane + 32 * t] = lane + 32 * t == j + 1 ? v1 : x[t];
      if (lane == 0) { e_out[j] = alpha; b_out[j] = beta; }
      __syncthreads();                                    // the product is there
#pragma unroll
      for (int t = 0; t < CS; ++t) { y[t] = ys[lane + 32 * t]; r[t] = rs[lane + 32 * t]; xy = fma(x[t], y[t], xy); }
      const double ya = ys[j + 1], ra = rs[j + 1], k0 = fma(alpha, fma(alpha, ra, -2.0 * ya), 0.0), u1 = fma(-alpha, ra, ya);
#pragma unroll
      for (int t = 0; t < CS; ++t) { y[t] = fma(-alpha, r[t], y[t]); us[lane + 32 * t] = y[t]; }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) xy += __shfl_xor_sync(0xFFFFFFFFu, xy, o);
      const double K2 = b2 * (xy + k0);
#pragma unroll
      for (int t = 0; t < CS; ++t) {
        const int c = lane + 32 * t;
        const double v = c == j + 1 ? v1 : x[t], p = -beta * v, qv = fma(-beta, y[t], K2 * v);
        pq[c] = make_double2(p, qv);
        x[t] = c > j + 1 ? fma(v1, qv, fma(u1, p, r[t])) : 0.0;
        xs[c] = x[t];
      }
      if (lane == 0) d_out[j + 1] = fma(-v1, fma(2.0 * beta, u1, -K2 * v1), ra);
      __syncthreads();                                    // the next update and the next column are there
    }
    if (lane == 0) e_out[n - 2] = xs[n - 1];
  }
}

// Eigenvalue and eigenvector number e (descending) of the tridiagonal matrix, one warp each (zt[e][.], normalised): multisection into 33 parts,
// a round costs 13 cycles per row (two points per lane: 24), twisted factorisation.  Behind them, one warp per panel of eight
// reflectors: H_8b ... H_8b+7 = I - V_b^T T_b V_b (T_b: inverse of diag(1 / beta) + the upper triangle of V_b V_b^T).
constexpr int WV_WARPS = 4, WV_ROUNDS = 7;                // of the multisection: relative width 2^-29
__global__ void __launch_bounds__(32 * WV_WARPS)
tridiag_vectors_kernel(const double* __restrict__ tri, const double* __restrict__ v, int n, double* __restrict__ zt, double* __restrict__ panels) {
  metis_pdl_wait_trigger();
  __shared__ __align__(16) double2 te[WT_MAX + 8];          // (a block beyond the matrix is read ahead)
  __shared__ double eo[WT_MAX + 1], dn[WV_WARPS][WT_MAX], up[WV_WARPS][WT_MAX];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
  const int n8 = (n + 7) & ~7, groups = (n + WV_WARPS - 1) / WV_WARPS;
  if ((int)blockIdx.x >= groups) {
    const int b = ((int)blockIdx.x - groups) * WV_WARPS + warp;
    if (8 * b + 2 >= n) return;
    double acc[2][2] = {};
    const bool on = 8 * b + g + 2 < n;
    const double* row = v + (int64_t)(on ? 8 * b + g : 0) * n;
#pragma unroll 4
    for (int kk = 0; kk < n8; kk += 8)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = kk + 4 * h + q;
        const double a = on && c < n ? row[c] : 0.0;
        metis_small::dmma(acc[h], a, a);                  // the fragments of V_b and of its transpose hold the same entries
      }
    double* t = dn[warp];
    t[8 * g + 2 * q] = acc[0][0] + acc[1][0]; t[8 * g + 2 * q + 1] = acc[0][1] + acc[1][1];
    __syncwarp();
    if (lane < 8) {
      double x[8];                                        // column `lane` of the lower triangular inverse: T_b transposed
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        double sum = 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) sum = fma(t[8 * i + k], x[k], sum);
        const double bt = 8 * b + i + 2 < n ? tri[2 * n + 8 * b + i] : 0.0;
        x[i] = i == lane ? bt : (i > lane ? -bt * sum : 0.0);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) panels[64 * b + 8 * lane + i] = x[i];        // T_b[lane][i]
    }
    return;
  }
  for (int i = tid; i <= n8; i += 32 * WV_WARPS) {
    const double e = i > 0 && i < n ? tri[n + i - 1] : 0.0;
    te[i] = i < n ? make_double2(tri[i], i > 0 ? fmax(e * e, metis_tri::TINY_SQUARE) : 0.0) : make_double2(4.0 * WT_MAX, 0.0);
    if (i > 0) eo[i - 1] = e;
  }
  __syncthreads();
  const int e = (int)blockIdx.x * WV_WARPS + warp;
  if (e >= n) return;
  double lm;
  {
    long long lo = __double_as_longlong(0x1p-56), hi = __double_as_longlong(2.0 * WT_MAX);
#pragma unroll 1
    for (int r = 0; r < WV_ROUNDS; ++r) {
      const long long w = (long long)((unsigned long long)(hi - lo + 32) / 33);
      const double x[1] = {__longlong_as_double(lo + w * (lane + 1))};
      int c[1];
      metis_tri::sturm_counts<1>(te, n8 >> 3, x, c);
      const unsigned int over = __ballot_sync(0xFFFFFFFFu, c[0] > n - 1 - e);
      const int f = over != 0u ? __ffs((int)over) - 1 : 32;
      hi = lo + w * (f + 1);
      lo += w * f;
    }
    lm = __longlong_as_double(lo + ((hi - lo) >> 1));
  }
  double *Dp = dn[warp], *Dm = up[warp];
  if (lane < 2) {                                         // pivots from the top and from the bottom
    double* D = lane ? Dm : Dp;
    double pm = 0.0, p = 1.0;
#pragma unroll 1
    for (int b = 0; b < n8; b += 8) {
      double d[8], e2[8];                                 // (rows beyond the matrix read padding, forwards, or row 0, backwards; nothing is kept)
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = b + u;
        d[u] = te[lane ? max(n - 1 - i, 0) : i].x - lm;
        e2[u] = te[lane ? max(n - i, 0) : i].y;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double pn = fma(d[u], p, -e2[u] * pm);
        d[u] = pn * metis_small::rcp_cubic(p + 1e-290);
        pm = p; p = pn;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = b + u;
        if (i < n) D[lane ? n - 1 - i : i] = d[u];
      }
      const int big = max(__double2hiint(p) & 0x7FF00000, __double2hiint(pm) & 0x7FF00000);
      const double sc = __hiloint2double(0x7FE00000 - big, 0);
      p *= sc; pm *= sc;
    }
  }
  __syncwarp();
  // twist where |gamma| is least: z = 1 there, the other entries are products of e / pivot outwards from it
  double best = 1e300;
  int at = 0;
  for (int i = lane; i < n; i += 32) {
    const double gamma = fabs(Dp[i] + Dm[i] - (te[i].x - lm));
    if (gamma < best) { best = gamma; at = i; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double other = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, at, o);
    if (other < best || (other == best && oi < at)) { best = other; at = oi; }
  }
  for (int i = lane; i < n; i += 32) {
    const double f = eo[i < at ? i : max(i - 1, 0)] * metis_small::rcp_cubic((i < at ? Dp[i] : Dm[i]) + 1e-60);
    Dm[i] = i == at ? 1.0 : -f;
  }
  __syncwarp();
  double zz = lane == 0 ? 1.0 : 0.0;
  if (lane < 2) {
    const int step = lane ? 1 : -1;
    double f = 1.0;
    for (int i = at + step; i >= 0 && i < n; i += 8 * step) {                  // eight at a time, the loads ahead of the products
      double m[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) { const int k = i + u * step; m[u] = k >= 0 && k < n ? Dm[k] : 0.0; }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int k = i + u * step;
        f *= m[u];
        zz = fma(f, f, zz);
        if (k >= 0 && k < n) Dm[k] = f;
      }
    }
  }
  __syncwarp();
  zz += __shfl_xor_sync(0xFFFFFFFFu, zz, 1);
  const double rz = metis_small::rsqrt_cubic(__shfl_sync(0xFFFFFFFFu, zz, 0));
  for (int i = lane; i < n; i += 32) zt[(int64_t)e * n + i] = Dm[i] * rz;
}

// x (n x n, column e: vector e, rows in the order of the factor's) = H_0 H_1 ... zt^T: eight vectors per CTA, panel by panel from the
// last, the sums over rows and then the rows dealt out to eight warps; the reflectors in shared memory.  Vectors beyond the
// factor's rank are zero.
constexpr int WB_WARPS = 8, WB_THREADS = 32 * WB_WARPS, WB_ZP = 12, WB_TILES = (WT_MAX / 8 + WB_WARPS - 1) / WB_WARPS;
__host__ __device__ constexpr size_t wb_smem(int n) { return sizeof(double) * (size_t)((n + 7) / 8 * 8) * ((n + 7) / 8 * 8 + 4 + WB_ZP); }
__global__ void __launch_bounds__(WB_THREADS)
tridiag_back_kernel(const double* __restrict__ zt, const double* __restrict__ v, const double* __restrict__ panels, const double* __restrict__ l,
                    const int* __restrict__ perm, int n, double* __restrict__ x) {
  metis_pdl_wait_trigger();
  extern __shared__ __align__(16) unsigned char wb_sm[];
  const int n8 = (n + 7) & ~7, P = n8 + 4;
  double* V = reinterpret_cast<double*>(wb_sm);           // [n8][P]
  double* Z = V + (size_t)n8 * P;                         // [n8][WB_ZP]: eight vectors as columns
  __shared__ double Ts[8 * WT_MAX];
  __shared__ __align__(16) double part[WB_WARPS][64], patch[64];               // stored in pairs
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, e0 = 8 * (int)blockIdx.x;
  const int n_panels = (n - 2 + 7) / 8;
  constexpr int CT = (WT_MAX + 31) / 32;
#pragma unroll 4
  for (int j = warp; j < n8; j += WB_WARPS) {
    double r[CT];
#pragma unroll
    for (int t = 0; t < CT; ++t) r[t] = j + 2 < n && lane + 32 * t < n ? v[(int64_t)j * n + lane + 32 * t] : 0.0;
#pragma unroll
    for (int t = 0; t < CT; ++t) if (lane + 32 * t < n8) V[j * P + lane + 32 * t] = r[t];
  }
  for (int o = tid; o < 64 * n_panels; o += WB_THREADS) Ts[o] = panels[o];
#pragma unroll
  for (int t = 0; t < CT; ++t) {                          // a warp per vector
    const int i = lane + 32 * t;
    if (i < n8) Z[i * WB_ZP + warp] = e0 + warp < n && i < n ? zt[(int64_t)(e0 + warp) * n + i] : 0.0;
  }
  const int rank = __syncthreads_count(tid < n && l[(int64_t)min(tid, n - 1) * (n + 1)] > 0.0);
  const int tiles = n8 / 8;
  for (int b = n_panels - 1; b >= 0; --b) {
    double acc[2][2] = {}, fa[WB_TILES][2], fb[WB_TILES][2];
#pragma unroll
    for (int u = 0; u < WB_TILES; ++u) {
      const int t = warp + WB_WARPS * u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        fa[u][h] = t < tiles ? V[(8 * b + g) * P + 8 * t + 4 * h + q] : 0.0;
        fb[u][h] = t < tiles ? Z[(8 * t + 4 * h + q) * WB_ZP + g] : 0.0;
      }
    }
#pragma unroll
    for (int u = 0; u < WB_TILES; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h) metis_small::dmma(acc[h], fa[u][h], fb[u][h]);
    *reinterpret_cast<double2*>(&part[warp][8 * g + 2 * q]) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
    // the update's operands, on the way meanwhile
    double d[WB_TILES][2];
#pragma unroll
    for (int u = 0; u < WB_TILES; ++u) {
      const int t = warp + WB_WARPS * u;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        fa[u][h] = t < tiles ? V[(8 * b + 4 * h + q) * P + 8 * t + g] : 0.0;
        d[u][h] = t < tiles ? Z[(8 * t + g) * WB_ZP + 2 * q + h] : 0.0;
      }
    }
    __syncthreads();
    if (warp == 0) {                                      // -T_b (V_b Z)
      double y[2] = {0.0, 0.0};
#pragma unroll
      for (int kk = 0; kk < 8; kk += 4) {
        const int at = 8 * (kk + q) + g;
        double sum = 0.0;
#pragma unroll
        for (int w = 0; w < WB_WARPS; ++w) sum += part[w][at];
        metis_small::dmma(y, Ts[64 * b + 8 * g + kk + q], sum);
      }
      *reinterpret_cast<double2*>(patch + 8 * g + 2 * q) = make_double2(-y[0], -y[1]);
    }
    __syncthreads();
    const double y0 = patch[8 * q + g], y1 = patch[8 * (q + 4) + g];
#pragma unroll
    for (int u = 0; u < WB_TILES; ++u) {
      const int t = warp + WB_WARPS * u;
      metis_small::dmma(d[u], fa[u][0], y0);
      metis_small::dmma(d[u], fa[u][1], y1);
      if (t < tiles) { Z[(8 * t + g) * WB_ZP + 2 * q] = d[u][0]; Z[(8 * t + g) * WB_ZP + 2 * q + 1] = d[u][1]; }
    }
    __syncthreads();
  }
  for (int o = tid; o < 8 * n; o += WB_THREADS) {
    const int i = o >> 3, e = o & 7;
    if (e0 + e < n) x[(int64_t)i * n + e0 + e] = e0 + e < rank ? Z[perm[i] * WB_ZP + e] : 0.0;
  }
}

// One product of a refinement step, 32 x 32 of the result per CTA (four warps of 16 x 16):
//   OP 0  W = L^T X      OP 1  S = W^T W (blockIdx.z = 0) and X^T X (blockIdx.z = 1)      OP 2  X' = X + X E
// Operands straight from L2 into fragment registers: n is at most 272 and each element is wanted by n / 32 CTAs.
template <int OP>
__global__ void __launch_bounds__(128)
refine_product_kernel(const double* __restrict__ a, const double* __restrict__ b, double* __restrict__ c, const double* __restrict__ a1,
                      double* __restrict__ c1, int n, const EigState* __restrict__ st, int step) {
  metis_pdl_wait_trigger();
  int last;
  if (eig_status(st, step, &last) != EIG_RUNNING) return;
  if (OP == 2 && eig_step_bad(st, step)) return;
  if (OP == 1 && blockIdx.z == 1) { a = a1; b = a1; c = c1; }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3;
  const int i0 = 32 * blockIdx.y + 16 * (warp & 1), j0 = 32 * blockIdx.x + 16 * (warp >> 1);
  double acc[2][2][2] = {};
  const bool in_i[2] = {i0 + g < n, i0 + 8 + g < n}, in_j[2] = {j0 + g < n, j0 + 8 + g < n};
  constexpr int U = 8;                                    // steps of four whose loads are in flight together
  for (int k0 = OP == 0 ? i0 / (4 * U) * (4 * U) : 0; k0 < n; k0 += 4 * U) {   // (L is lower triangular)
    double fa[U][2], fb[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + 4 * u + q;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        fa[u][h] = k < n && in_i[h] ? __ldcg(OP == 2 ? a + (int64_t)(i0 + 8 * h + g) * n + k : a + (int64_t)k * n + i0 + 8 * h + g) : 0.0;
        fb[u][h] = k < n && in_j[h] ? __ldcg(b + (int64_t)k * n + j0 + 8 * h + g) : 0.0;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int v = 0; v < 2; ++v) metis_small::dmma(acc[h][v], fa[u][h], fb[u][v]);
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int i = i0 + 8 * h + g, j = j0 + 8 * v + 2 * q + e;
        if (i < n && j < n) c[(int64_t)i * n + j] = acc[h][v][e] + (OP == 2 ? a[(int64_t)i * n + j] : 0.0);
      }
}

// E of a step from S and G1 = X^T X, and what the status is made of
__global__ void __launch_bounds__(256)
refine_correction_kernel(const double* __restrict__ s, const double* __restrict__ g1, double* __restrict__ e_out, int n, EigState* __restrict__ st, int step) {
  metis_pdl_wait_trigger();
  int last;
  if (eig_status(st, step, &last) != EIG_RUNNING) return;
  const int o = blockIdx.x * 256 + threadIdx.x;
  float em = 0.0f, en = 0.0f;
  bool open = false;
  if (o < n * n) {
    const int i = o / n, j = o % n;
    const double gi = g1[(int64_t)i * n + i], gj = g1[(int64_t)j * n + j];
    double e = 0.0;
    if (gi != 0.0 && gj != 0.0) {                         // zero columns stay
      const double r = (i == j ? 1.0 : 0.0) - g1[o];
      e = 0.5 * r;
      if (i != j) {
        const double sv = s[o], li = s[(int64_t)i * n + i] / gi, lj = s[(int64_t)j * n + j] / gj;
        const double ro = 0.5 * r * (li + lj);            // what orthonormalising alone adds to S_ij
        if (fmax(sv * sv, ro * ro) > 1e-28 * fabs(li * lj)) {                      // orthogonal to FP64 rounding otherwise, and stays so
          const double gap = lj - li, a = sv + lj * r, b = sv + li * r;
          if (fabs(a) < 0.0625 * fabs(gap) && fabs(b) < 0.0625 * fabs(gap)) e = a / gap;
          else if (sv * sv > 1e-24 * fabs(li * lj)) open = true;
        }
      }
    }
    e_out[o] = e;
    em = fabsf((float)e);
    en = em * em;
  }
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) { em = fmaxf(em, __shfl_xor_sync(0xFFFFFFFFu, em, d)); en += __shfl_xor_sync(0xFFFFFFFFu, en, d); }
  const bool any = __any_sync(0xFFFFFFFFu, open);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&st->emax[step], __float_as_uint(em));
    atomicAdd(&st->norm2[step], eig_norm2_units(en));
    if (any) st->open[step] = 1;
  }
}

// eigenvalues descending (squared lengths of the last step's S), eigenvectors in the input's row order
__global__ void __launch_bounds__(1024, 1)
eigen_finish_kernel(const double* __restrict__ x0, const double* __restrict__ x1, const double* __restrict__ s, const double* __restrict__ g1,
                    const int* __restrict__ perm, int n, const EigState* __restrict__ st, double* __restrict__ evals, double* __restrict__ evecs,
                    int* __restrict__ failed) {
  metis_pdl_wait_trigger();
  __shared__ double lam[MAXQ_WIDE];
  __shared__ int order[MAXQ_WIDE];
  int last;
  const bool done = eig_status(st, ER_STEPS, &last) == EIG_DONE;
  const int tid = threadIdx.x;
  if (tid == 0) *failed = done ? 0 : 1;
  if (!done) return;
  const double* x = last & 1 ? x0 : x1;                   // step t reads one buffer and writes the other
  if (tid < n) {
    const double gi = g1[(int64_t)tid * n + tid];
    lam[tid] = gi > 0.0 ? s[(int64_t)tid * n + tid] / gi : 0.0;
    order[tid] = tid;
  }
  __syncthreads();
  if (tid < n) {
    const double li = lam[tid];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += (lam[j] > li) || (lam[j] == li && j < tid);
    order[rank] = tid;                                    // stays a valid index if NaNs make ranks collide
  }
  __syncthreads();
  if (tid < n) evals[tid] = lam[order[tid]];
  for (int o = tid; o < n * n; o += 1024) {
    const int i = o / n, t = o % n;
    evecs[(int64_t)perm[i] * n + t] = x[(int64_t)i * n + order[t]];
  }
}

// ------------------------------------------------------------------------------------------------
// One-sided (Hestenes) Jacobi on the columns of Y = L (the Cholesky factor of the Gram matrix, so that
// G = Y Y^T and the rotated columns end as U Sigma), for n up to MAXQ_WIDE, on ONE CLUSTER of JC_P CTAs.
// The 2 * JC_P * JC_W column slots are dealt out as 2 * JC_P blocks of JC_W columns; every CTA holds two blocks in
// its shared memory (FP64, 78 KB) and orthogonalises, one warp per couple,
//   - in the first outer round of a sweep: every pair among its 2 * JC_W columns (round-robin tournament),
//   - in the other outer rounds: every pair of one column of each block,
// then the blocks move on to the neighbouring CTAs in the order of a round-robin tournament over blocks (block 0
// stays), written straight into the neighbour's second buffer through distributed shared memory, between two
// cluster barriers.  After 2 * JC_P - 1 outer rounds every pair of columns has met once: one sweep.  Arithmetic of
// a rotation as in the one-CTA solver: columns and rotation orthonormality in FP64, steering quantities in FP32.
constexpr int JC_P = 8, JC_W = 17, JC_ROWS = 288, JC_THREADS = 32 * JC_W;
constexpr int JC_RL = JC_ROWS / 32;                     // rows per lane
constexpr size_t JC_SMEM = sizeof(double) * 2 * 2 * JC_W * JC_ROWS;

// Rotation that makes two columns with squared norms a, b and inner product c orthogonal: the smaller root of
// tan(2 theta) = 2c / (b - a), |theta| <= pi / 4.  The FP32 quantities only steer convergence (fast reciprocal square
// roots); (cs, sn) is made a unit vector to ~1e-14 by one Newton step in FP64; tf = tan(theta) updates the carried norms.
__device__ __forceinline__ void jc_rotation(float a, float b, float cf, double& cs, double& sn, float& tf) {
  const float d = b - a, c2 = 2.0f * cf;
  const float h2 = fmaf(c2, c2, d * d);
  const float rh = rsqrtf(h2);
  const float cc = fmaf(0.5f * fabsf(d), rh, 0.5f);
  const float rs = rsqrtf(cc);
  const float c32 = cc * rs, s32 = (d < 0.0f ? -c2 : c2) * (0.5f * rh) * rs;
  tf = s32 * rs;
  const double cd = (double)c32, sd = (double)s32;
  const double scale = 1.5 - 0.5 * (cd * cd + sd * sd);
  cs = cd * scale; sn = sd * scale;
}

__global__ void __cluster_dims__(JC_P, 1, 1) __launch_bounds__(JC_THREADS, 1)
jacobi_cluster_kernel(const double* __restrict__ l, int n, float exit_cos2, const int* __restrict__ wanted, double* __restrict__ ycm) {
  if (!*wanted) return;                                   // the same for every CTA of the cluster
  extern __shared__ __align__(16) unsigned char jsm[];
  double* cols = reinterpret_cast<double*>(jsm);        // [buffer][slot][column][row]
  __shared__ float nrm[2][JC_W];
  __shared__ int flag_s;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  auto col_ptr = [&](int buf, int slot, int c) { return cols + (((size_t)buf * 2 + slot) * JC_W + c) * JC_ROWS; };
  // load: slot s of this CTA starts as block 2 * rank + s, i.e. columns (2 * rank + s) * JC_W + c of Y
  for (int o = tid; o < 2 * JC_W * JC_ROWS; o += JC_THREADS) {
    const int i = o % JC_ROWS, c = (o / JC_ROWS) % JC_W, s = o / (JC_ROWS * JC_W);
    const int gc = (2 * rank + s) * JC_W + c;
    col_ptr(0, s, c)[i] = (gc < n && i < n && gc <= i) ? l[(int64_t)i * n + gc] : 0.0;
  }
  __syncthreads();
  int cur = 0;
  for (int sweep = 0; sweep < 16; ++sweep) {
    bool above = false;
    int any_above = 0;
    for (int orr = 0; orr < 2 * JC_P - 1; ++orr) {
      // exact norms of this CTA's columns at the start of every outer round (they are carried through the rounds)
      for (int sc = warp; sc < 2 * JC_W; sc += JC_W) {
        const double* y = col_ptr(cur, sc / JC_W, sc % JC_W);
        double a = 0.0;
#pragma unroll
        for (int t = 0; t < JC_RL; ++t) { const double v = y[lane + 32 * t]; a += v * v; }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
        if (lane == 0) nrm[sc / JC_W][sc % JC_W] = (float)a;
      }
      __syncthreads();
      if (orr == 0) {
        // every pair among the CTA's 2 * JC_W columns: round-robin tournament, both columns of a couple through shared memory
        for (int r = 0; r < 2 * JC_W - 1; ++r) {
          int p, q;
          jc_pair(warp, r, 2 * JC_W, &p, &q);
          const int ps = p / JC_W, pc = p % JC_W, qs = q / JC_W, qc = q % JC_W;
          double* yp_s = col_ptr(cur, ps, pc);
          double* yq_s = col_ptr(cur, qs, qc);
          double yp[JC_RL], yq[JC_RL];
          double c = 0.0;
#pragma unroll
          for (int t = 0; t < JC_RL; ++t) { yp[t] = yp_s[lane + 32 * t]; yq[t] = yq_s[lane + 32 * t]; c += yp[t] * yq[t]; }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
          const float a = nrm[ps][pc], b = nrm[qs][qc], cf = (float)c;
          if (cf * cf > 1e-26f * (a * b)) {
            double cs, sn; float tf;
            jc_rotation(a, b, cf, cs, sn, tf);
#pragma unroll
            for (int t = 0; t < JC_RL; ++t) {
              yp_s[lane + 32 * t] = cs * yp[t] - sn * yq[t];
              yq_s[lane + 32 * t] = sn * yp[t] + cs * yq[t];
            }
            const float tc = tf * cf;
            if (lane == 0) { nrm[ps][pc] = a - tc; nrm[qs][qc] = b + tc; }
            above |= cf * cf > exit_cos2 * (a * b);
          }
          __syncthreads();
        }
      } else {
        // every pair of one column of each block: warp w keeps column w of the first block in registers for all
        // JC_W rounds (nobody else touches it) and meets the columns of the second block one after the other
        double* yp_s = col_ptr(cur, 0, warp);
        double yp[JC_RL];
#pragma unroll
        for (int t = 0; t < JC_RL; ++t) yp[t] = yp_s[lane + 32 * t];
        float a = nrm[0][warp];
        for (int r = 0; r < JC_W; ++r) {
          const int qc = (warp + r) % JC_W;
          double* yq_s = col_ptr(cur, 1, qc);
          double yq[JC_RL];
          double c = 0.0;
#pragma unroll
          for (int t = 0; t < JC_RL; ++t) { yq[t] = yq_s[lane + 32 * t]; c += yp[t] * yq[t]; }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
          const float b = nrm[1][qc], cf = (float)c;
          if (cf * cf > 1e-26f * (a * b)) {
            double cs, sn; float tf;
            jc_rotation(a, b, cf, cs, sn, tf);
#pragma unroll
            for (int t = 0; t < JC_RL; ++t) {
              const double np_ = cs * yp[t] - sn * yq[t];
              yq_s[lane + 32 * t] = sn * yp[t] + cs * yq[t];
              yp[t] = np_;
            }
            const float tc = tf * cf;
            above |= cf * cf > exit_cos2 * (a * b);
            if (lane == 0) nrm[1][qc] = b + tc;
            a -= tc;
          }
          __syncthreads();
        }
#pragma unroll
        for (int t = 0; t < JC_RL; ++t) yp_s[lane + 32 * t] = yp[t];
        __syncthreads();
      }
      const bool last = orr == 2 * JC_P - 2;
      if (last) {
        const int any = __syncthreads_or(above ? 1 : 0);
        if (tid == 0) flag_s = any;
      }
      cluster.sync();                                    // every CTA is done with this outer round (flags are written)
      // hand the blocks on: slot 0 ("top") of CTA c goes to the top of c + 1 (the last CTA's top becomes its own
      // bottom, CTA 0's top stays); slot 1 ("bottom") of CTA c goes to the bottom of c - 1 (CTA 0's bottom becomes
      // the top of CTA 1)
      {
        int dst_rank[2], dst_slot[2];
        if (rank == 0) { dst_rank[0] = 0; dst_slot[0] = 0; dst_rank[1] = 1; dst_slot[1] = 0; }
        else {
          if (rank == JC_P - 1) { dst_rank[0] = rank; dst_slot[0] = 1; } else { dst_rank[0] = rank + 1; dst_slot[0] = 0; }
          dst_rank[1] = rank - 1; dst_slot[1] = 1;
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const double2* src = reinterpret_cast<const double2*>(col_ptr(cur, s, 0));
          double2* dst = reinterpret_cast<double2*>(cluster.map_shared_rank(col_ptr(cur ^ 1, dst_slot[s], 0), dst_rank[s]));
          for (int o = tid; o < JC_W * JC_ROWS / 2; o += JC_THREADS) dst[o] = src[o];
        }
      }
      if (last) {
        for (int c = 0; c < JC_P; ++c) any_above |= *cluster.map_shared_rank(&flag_s, c);
      }
      cluster.sync();                                    // the blocks have landed; the flags have been read
      cur ^= 1;
    }
    if (!any_above) break;
  }
  // column-major result: ycm[(slot position) * n + row]; the order of the columns is irrelevant (they are sorted
  // by their norms afterwards)
  for (int o = tid; o < 2 * JC_W * n; o += JC_THREADS) {
    const int i = o % n, sc = o / n;
    ycm[((int64_t)(2 * rank) * JC_W + sc) * n + i] = col_ptr(cur, sc / JC_W, sc % JC_W)[i];
  }
}

// eigenvalues = squared column norms (descending), eigenvectors = normalised columns: evecs[i * n + t]
__global__ void __launch_bounds__(1024, 1)
jacobi_collect_kernel(const double* __restrict__ ycm, int n, const int* __restrict__ perm, const int* __restrict__ wanted, double* __restrict__ evals,
                      double* __restrict__ evecs) {
  if (!*wanted) return;
  constexpr int NC = 2 * JC_P * JC_W;
  __shared__ double lam[NC];
  __shared__ int order[NC];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int c = warp; c < NC; c += 32) {
    double a = 0.0;
    for (int i = lane; i < n; i += 32) { const double v = ycm[(int64_t)c * n + i]; a += v * v; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    if (lane == 0) { lam[c] = a; order[c] = c; }
  }
  __syncthreads();
  if (tid < NC) {
    const double li = lam[tid];
    int rank = 0;
    for (int j = 0; j < NC; ++j) rank += (lam[j] > li) || (lam[j] == li && j < tid);
    order[rank] = tid;                                  // stays a valid index if NaNs make ranks collide
  }
  __syncthreads();
  if (tid < n) evals[tid] = lam[order[tid]];
  for (int o = tid; o < n * n; o += 1024) {
    const int i = o / n, t = o % n;
    const int c = order[t];
    const double l2 = lam[c];
    evecs[(int64_t)perm[i] * n + t] = l2 > 0.0 ? ycm[(int64_t)c * n + i] * (1.0 / sqrt(l2)) : 0.0;
  }
}

// ------------------------------------------------------------------------------------------------
// Sign convention, one CTA per factor vector j: the entry of largest magnitude of right[j][:] (lowest index on ties)
// is made positive; sign[j] records the flip for the left factor; amax|right| into *amax_out.
__global__ void __launch_bounds__(256)
sign_rows_kernel(float* __restrict__ right, int64_t cols, float* __restrict__ sign_out, float* __restrict__ amax_out) {
  metis_pdl_wait_trigger();
  __shared__ float bv[8], bs_[8];
  __shared__ int bi[8];
  __shared__ float sg_s;
  const int j = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* row = right + (int64_t)j * cols;
  float av = -1.0f, sv = 0.0f;
  int ai = 0x7FFFFFFF;
  for (int64_t c = tid; c < cols; c += 256) {
    const float v = row[c];
    if (fabsf(v) > av) { av = fabsf(v); sv = v; ai = (int)c; }      // increasing c: the first maximum is kept
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xFFFFFFFFu, av, o), os = __shfl_xor_sync(0xFFFFFFFFu, sv, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, ai, o);
    if (ov > av || (ov == av && oi < ai)) { av = ov; sv = os; ai = oi; }
  }
  if (lane == 0) { bv[warp] = av; bs_[warp] = sv; bi[warp] = ai; }
  __syncthreads();
  if (tid == 0) {
    for (int w = 1; w < 8; ++w)
      if (bv[w] > bv[0] || (bv[w] == bv[0] && bi[w] < bi[0])) { bv[0] = bv[w]; bs_[0] = bs_[w]; bi[0] = bi[w]; }
    const float sg = bs_[0] < 0.0f ? -1.0f : 1.0f;
    sg_s = sg;
    sign_out[j] = sg;
    if (amax_out != nullptr) atomicMax(reinterpret_cast<unsigned int*>(amax_out), __float_as_uint(fmaxf(bv[0], 0.0f)));
  }
  __syncthreads();
  if (sg_s < 0.0f)
    for (int64_t c = tid; c < cols; c += 256) row[c] = -row[c];
}

// ------------------------------------------------------------------------------------------------
// coef[r][j0 + jj] = sum over slices s of part[s][r][jj]  (jj < gw, fixed order), and the BF16 terms of those
// coefficients in the residual product's A operand: a6[r][term * kp + j0 + jj], terms [h | h | l | h | l2 | l].
// One thread per (row, group of eight columns).  The group with j0 == 0 also clears the padding of a6 beyond 6 kp.
__global__ void __launch_bounds__(256)
coef_sum_kernel(const float* __restrict__ part, int slices, int64_t rows, int gw, int j0, int kp, float* __restrict__ coef,
                __nv_bfloat16* __restrict__ a6, int kx) {
  metis_pdl_wait_trigger();
  const int g8 = gw / 8;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= rows * g8) return;
  const int64_t r = idx / g8;
  const int jj = (int)(idx % g8) * 8;
  float v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) v[e] = 0.0f;
  for (int s = 0; s < slices; ++s) {
    const float4 p0 = *reinterpret_cast<const float4*>(part + ((int64_t)s * rows + r) * gw + jj);
    const float4 p1 = *reinterpret_cast<const float4*>(part + ((int64_t)s * rows + r) * gw + jj + 4);
    v[0] += p0.x; v[1] += p0.y; v[2] += p0.z; v[3] += p0.w; v[4] += p1.x; v[5] += p1.y; v[6] += p1.z; v[7] += p1.w;
  }
  float* cd = coef + r * kp + j0 + jj;
  *reinterpret_cast<float4*>(cd) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(cd + 4) = make_float4(v[4], v[5], v[6], v[7]);
  if (a6 != nullptr) {
    uint4 h, l, l2;
    metis_split3x8(v, h, l, l2);
    __nv_bfloat16* dst = a6 + r * kx + j0 + jj;
    *reinterpret_cast<uint4*>(dst) = h; *reinterpret_cast<uint4*>(dst + kp) = h; *reinterpret_cast<uint4*>(dst + 2 * kp) = l;
    *reinterpret_cast<uint4*>(dst + 3 * kp) = h; *reinterpret_cast<uint4*>(dst + 4 * kp) = l2; *reinterpret_cast<uint4*>(dst + 5 * kp) = l;
    if (j0 == 0 && jj == 0)
      for (int z = 6 * kp; z < kx; z += 8) *reinterpret_cast<uint4*>(a6 + r * kx + z) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// gathers the sampled rows of x into a contiguous matrix: xs[j][:] = x[idx[j]][:]   (16 bytes per thread)
__global__ void __launch_bounds__(256)
gather_rows_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, const int* __restrict__ idx, int n_s, __nv_bfloat16* __restrict__ xs) {
  metis_pdl_wait_trigger();
  const int64_t per_row = cols / 8;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= (int64_t)n_s * per_row) return;
  const int64_t j = i / per_row, c8 = i % per_row;
  reinterpret_cast<uint4*>(xs)[i] = reinterpret_cast<const uint4*>(x + (int64_t)idx[j] * cols)[c8];
}

}  // namespace metis_wide
