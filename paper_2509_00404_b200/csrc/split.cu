// Low-rank + residual split of one GEMM operand (Sections 3.1 and 3.2) and its NVFP4 quantization.
//
// Steps (FULL = on all rows, SAMPLED = subspace from a sparse row sample, "broadcast" to all rows):
//   amax(x) -> row sample -> sketch Z = x[S,:] Omega (Omega from Philox + quantile table, never stored)
//   -> CholeskyQR2 (FP64 Gram + Cholesky) -> M = H^T x[S,:] -> eigen-decomposition of M M^T (Jacobi
//   sweeps in FP32, refined in FP64) -> right basis B -> [SAMPLED: C = x B, Rayleigh-Ritz on C^T C] -> residual R = x - C B^T fused
//   with the NVFP4 quantizer in both block orientations -> factor rotation, sign fix, factor quantization.
#include "quant_tile.cuh"
#include "bigrank.cuh"
#include "small_eig.cuh"

metis_status_t metis_launch_residual_tc(metis_context* ctx, const void* x, const float* coef, int k, int kp,
                                        const metis_qt::QuantParams& qp, const float* amax_src, float* ts_out0, float* ts_out1,
                                        float* dense, void* a6, void* b6, cudaStream_t s);

namespace {

constexpr int MAXQ = metis_small::MAXQ;                // k + p at most (k = 64 with p = 8)
constexpr int LP = metis_small::PITCH;                 // row pitch of a factor in shared memory

// ------------------------------------------------------------------------------------------------
// The sampled rows; the first block of the one-CTA chain's call also clears what its later kernels accumulate into (a memset of
// its own was a launch in front of every decomposition).
__global__ void sample_rows_kernel(int* __restrict__ idx, int n_s, int64_t rows, uint64_t seed, int full, float* __restrict__ amax, unsigned long long* __restrict__ keys) {
  metis_pdl_wait_trigger();
  if (blockIdx.x == 0 && amax != nullptr && threadIdx.x < 64) {
    if (threadIdx.x < 16) amax[threadIdx.x] = 0.0f;
    keys[threadIdx.x] = 0ull;
  }
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_s) return;
  if (full) { idx[j] = j; return; }
  const uint32_t g = (uint32_t)(rows / n_s);
  const uint4 w = metis_philox((uint32_t)j, 0u, METIS_STREAM_SAMPLING, 0u, (uint32_t)seed, (uint32_t)(seed >> 32));
  idx[j] = (int)((uint32_t)j * g + w.x % g);          // one row per stratum of g consecutive rows
}

// ------------------------------------------------------------------------------------------------
// Device-detected conditions of a split: amax|x| not finite (a NaN or an infinity in the operand: amax is kept as
// an ordered bit pattern, so a NaN ranks above every number), a non-finite eigenvalue.  One warp.
__global__ void split_status_kernel(const float* __restrict__ amax, const double* __restrict__ evals, int k, uint32_t* dev_status) {
  metis_pdl_wait_trigger();
  uint32_t bits = 0u;
  if (threadIdx.x == 0 && !(fabsf(*amax) <= 3.0e38f)) bits |= METIS_DEV_NONFINITE;
  for (int j = threadIdx.x; j < k; j += 32)
    if (!(fabs(evals[j]) <= 1.0e300)) bits |= METIS_DEV_NUMERIC;
  if (bits) atomicOr(dev_status, bits);
}

__global__ void reduce_partials_kernel(const float* __restrict__ zp, int n_chunks, int64_t n, float* __restrict__ z) {
  metis_pdl_wait_trigger();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float acc = 0.0f;
  int c = 0;
  for (; c + 8 <= n_chunks; c += 8) {                                    // eight loads in flight; fixed order: reproducible
    float t[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) t[u] = zp[(int64_t)(c + u) * n + i];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc += t[u];
  }
  for (; c < n_chunks; ++c) acc += zp[(int64_t)c * n + i];
  z[i] = acc;
}

// ------------------------------------------------------------------------------------------------
// Gram partials in FP64: part[p][i][j] = sum over the p-th slab of rows r of v(r,i) v(r,j),
// v(r,i) = V[r*stride_row + i*stride_vec].
// On the FP64 tensor cores: 64 rows at a time are converted to FP64 in shared memory (FP32 -> FP64 conversions are a slow-rate
// instruction: once per element), a warp owns up to six lower 8 x 8 tiles of the result.  As FP64 multiply-adds
// from shared memory the same slabs took 8.4 us (4096 x 40) and 24 us (16384 x 40).
constexpr int GR_TILE = 64;
constexpr int GR_TPW = 6;                               // tiles per warp: 45 lower tiles at n = 72 over eight warps
__global__ void __launch_bounds__(256)
gram_kernel(const float* __restrict__ v, int64_t n_rows, int n, int64_t stride_row, int64_t stride_vec,
            int64_t rows_per_part, double* __restrict__ part, const int* __restrict__ skip) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;                 // second CholeskyQR pass not needed (see chol_kernel)
  __shared__ double tile[GR_TILE][LP];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q4 = lane & 3;
  const int64_t r_begin = (int64_t)blockIdx.x * rows_per_part;
  const int64_t r_end = min(n_rows, r_begin + rows_per_part);
  const int n8 = (n + 7) & ~7, tiles = (n8 / 8) * (n8 / 8 + 1) / 2;
  int t_i[GR_TPW], t_j[GR_TPW];
  double acc[GR_TPW][2][2];                             // even and odd steps: two chains in flight
#pragma unroll
  for (int u = 0; u < GR_TPW; ++u) {
    const int o = warp + 8 * u;
    int ti = 0;
    while ((ti + 1) * (ti + 2) / 2 <= o) ++ti;
    t_i[u] = ti; t_j[u] = o - ti * (ti + 1) / 2;
    acc[u][0][0] = acc[u][0][1] = acc[u][1][0] = acc[u][1][1] = 0.0;
  }
  for (int i = tid; i < GR_TILE * (n8 - n); i += 256) tile[i / (n8 - n)][n + i % (n8 - n)] = 0.0;
  for (int64_t r0 = r_begin; r0 < r_end; r0 += GR_TILE) {
    if (stride_row == 1) {
      for (int i = tid; i < GR_TILE * n; i += 256) {
        const int rr = i % GR_TILE, ii = i / GR_TILE;
        tile[rr][ii] = r0 + rr < r_end ? (double)v[r0 + rr + ii * stride_vec] : 0.0;
      }
    } else {
      for (int i = tid; i < GR_TILE * n; i += 256) {
        const int ii = i % n, rr = i / n;
        tile[rr][ii] = r0 + rr < r_end ? (double)v[(r0 + rr) * stride_row + ii * stride_vec] : 0.0;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < GR_TPW; ++u) {
      if (warp + 8 * u < tiles) {
        const double* pa = &tile[q4][8 * t_i[u] + g];
        const double* pb = &tile[q4][8 * t_j[u] + g];
#pragma unroll
        for (int kk = 0; kk < GR_TILE; kk += 8) {
          metis_small::dmma(acc[u][0], pa[kk * LP], pb[kk * LP]);
          metis_small::dmma(acc[u][1], pa[(kk + 4) * LP], pb[(kk + 4) * LP]);
        }
      }
    }
    __syncthreads();
  }
  double* out = part + (int64_t)blockIdx.x * n * n;
#pragma unroll
  for (int u = 0; u < GR_TPW; ++u) {
    if (warp + 8 * u < tiles) {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int i = 8 * t_i[u] + g, j = 8 * t_j[u] + 2 * q4 + e;
        const double x = acc[u][0][e] + acc[u][1][e];
        if (i < n && j < n) {
          out[i * n + j] = x;
          if (t_i[u] != t_j[u]) out[j * n + i] = x;
        }
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------
// One CholeskyQR pass, step 1 (one CTA): G = L L^T in FP64; writes L^-T (q x q, row-major, zero below the diagonal), so that step 2
// is a product on many CTAs instead of a triangular solve per row.  A pivot below 1e-13 of the largest diagonal marks a
// dependent sketch column: the corresponding column of H = Z L^-T becomes zero instead of amplified noise.
constexpr size_t CHOL_SMEM = sizeof(double) * MAXQ * LP;
__global__ void __launch_bounds__(512)
chol_kernel(const double* __restrict__ g, int q, double* __restrict__ linvt_out, const int* __restrict__ skip, int* __restrict__ well_conditioned) {
  metis_pdl_wait();
  if (skip != nullptr && *skip) return;
  extern __shared__ __align__(16) double xs[];
  __shared__ double L[MAXQ][LP];
  __shared__ double gmax_s;
  __shared__ double dmin_s;
  __shared__ double inv_s[MAXQ];
  const int tid = threadIdx.x, q8 = (q + 7) & ~7;
  for (int o = tid; o < q8 * q8; o += 512) {
    const int i = o / q8, j = o % q8;
    L[i][j] = i < q && j < q ? g[i * q + j] : 0.0;
  }
  __syncthreads();
  if (tid < 32) {
    double gm = 0.0;
    for (int i = tid; i < q; i += 32) gm = fmax(gm, L[i][i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) gm = fmax(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, o));
    if (tid == 0) gmax_s = gm;
  }
  __syncthreads();
  const double tol = 1e-13 * gmax_s;
  metis_small::cta_cholesky<LP>(&L[0][0], q, tol, inv_s, &dmin_s, 512);
  // With every pivot above 1e-8 of the largest diagonal the FP64 factorisation leaves Z L^-T orthonormal to
  // ~1e-8 already, below the FP32 rounding of its storage: the caller's second pass is then skipped.
  metis_pdl_trigger();
  if (tid == 0 && well_conditioned != nullptr) *well_conditioned = (dmin_s > 1e-8 * gmax_s) ? 1 : 0;
  metis_small::cta_invert_lower<LP>(&L[0][0], inv_s, q, xs, LP, 512);
  for (int o = tid; o < q * q; o += 512) { const int i = o / q, j = o % q; linvt_out[o] = i <= j ? xs[j * LP + i] : 0.0; }
}

// One CholeskyQR pass, steps 0 and 1 in one CTA, for a sketch short enough to sit in shared memory as FP64 (the
// row-sampled case: a few hundred rows): G = Z^T Z and its Cholesky factor without a trip through global memory.
// The Gram matrix is formed on the FP64 tensor cores, a warp per lower 8 x 8 tile (as FP64 multiply-adds from shared memory
// it took half of the kernel: 22 -> 9 us at 160 x 40 with the panel factorisation).
constexpr int GC_THREADS = 512;
constexpr size_t GC_MAX_SMEM = 176 * 1024;              // beside ~45 KiB of static shared memory: 288 sampled rows at q = 72
__host__ __device__ inline int gram_chol_pitch(int q) { return ((q + 7) & ~7) + 4; }   // 4 or 12 mod 16: conflict-free fragment loads
__host__ inline size_t gram_chol_smem(int64_t n_s, int q) { return (size_t)n_s * gram_chol_pitch(q) * sizeof(double); }
// Well-conditioned sketch (every pivot above 1e-8 of the largest diagonal: Z L^-T is orthonormal to ~1e-8 already):
// the kernel writes L^-T and clears *applied; orth_apply_kernel, on many CTAs, multiplies by it.  Otherwise (rare) the whole CholeskyQR2 runs here on the FP64 copy - solve, second Gram
// matrix, second factor, second solve - H is written over z and *applied is set, which makes the apply kernel
// behind this one return at once.
__global__ void __launch_bounds__(GC_THREADS, 1)
gram_chol_kernel(float* __restrict__ z, int n_s, int q, double* __restrict__ linvt_out, int* __restrict__ applied) {
  metis_pdl_wait();
  extern __shared__ __align__(16) double zs[];
  __shared__ double L[MAXQ][LP];
  __shared__ double gmax_s;
  __shared__ double dmin_s;
  __shared__ double inv_s[MAXQ];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q8 = (q + 7) & ~7, zp = gram_chol_pitch(q);
  for (int o = tid; o < n_s * zp; o += GC_THREADS) {
    const int r = o / zp, c = o - r * zp;
    zs[o] = c < q ? (double)z[(int64_t)r * q + c] : 0.0;
  }
  const int g = lane >> 2, q4 = lane & 3, tiles = (q8 / 8) * (q8 / 8 + 1) / 2;
  bool solved_here = false;
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
    for (int o = warp; o < tiles; o += GC_THREADS / 32) {
      int ti = 0;
      while ((ti + 1) * (ti + 2) / 2 <= o) ++ti;
      const int tj = o - ti * (ti + 1) / 2;
      double acc[4][2] = {};
      const double* pa = zs + q4 * zp + 8 * ti + g;
      const double* pb = zs + q4 * zp + 8 * tj + g;
      for (int r0 = 0; r0 < n_s; r0 += 16) {               // n_s is a multiple of 16
#pragma unroll
        for (int u = 0; u < 4; ++u) metis_small::dmma(acc[u], pa[(r0 + 4 * u) * zp], pb[(r0 + 4 * u) * zp]);
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) L[8 * ti + g][8 * tj + 2 * q4 + e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
    }
    __syncthreads();
    if (tid < 32) {
      double gm = 0.0;
      for (int i = tid; i < q; i += 32) gm = fmax(gm, L[i][i]);
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) gm = fmax(gm, __shfl_xor_sync(0xFFFFFFFFu, gm, off));
      if (tid == 0) gmax_s = gm;
    }
    __syncthreads();
    const double tol = 1e-13 * gmax_s;
    metis_small::cta_cholesky<LP>(&L[0][0], q, tol, inv_s, &dmin_s, GC_THREADS);
    metis_pdl_trigger();
    if (pass == 0 && dmin_s > 1e-8 * gmax_s) break;
    // z_row <- z_row L^-T in shared memory by forward substitution, one warp per row, column-oriented: lane i % 32 keeps z_i; step j
    // broadcasts h_j = z_j / L[j][j] from its owner and every lane subtracts h_j L[i][j] from its own later entries
    solved_here = true;
    for (int r = warp; r < n_s; r += GC_THREADS / 32) {
      double* zr = zs + r * zp;
      double z0 = lane < q ? zr[lane] : 0.0, z1 = lane + 32 < q ? zr[lane + 32] : 0.0, z2 = lane + 64 < q ? zr[lane + 64] : 0.0;
      for (int j = 0; j < q; ++j) {
        const double lj0 = lane < q ? L[lane][j] : 0.0;
        const double lj1 = lane + 32 < q ? L[lane + 32][j] : 0.0;
        const double lj2 = lane + 64 < q ? L[lane + 64][j] : 0.0;
        const double zj = __shfl_sync(0xFFFFFFFFu, j < 32 ? z0 : (j < 64 ? z1 : z2), j & 31);
        const double hj = zj * inv_s[j];
        if (lane == (j & 31)) { if (j < 32) z0 = hj; else if (j < 64) z1 = hj; else z2 = hj; }
        if (lane > j) z0 -= hj * lj0;
        if (lane + 32 > j) z1 -= hj * lj1;
        if (lane + 64 > j) z2 -= hj * lj2;
      }
      if (lane < q) zr[lane] = z0;
      if (lane + 32 < q) zr[lane + 32] = z1;
      if (lane + 64 < q) zr[lane + 64] = z2;
    }
    __syncthreads();
  }
  if (tid == 0) *applied = solved_here ? 1 : 0;
  if (solved_here) {
    for (int e = tid; e < n_s * q; e += GC_THREADS) z[e] = (float)zs[(e / q) * zp + e % q];
  } else {
    // the FP64 copy of z is not needed any more: n_s >= q rows of the same pitch hold the inverse
    metis_small::cta_invert_lower<LP>(&L[0][0], inv_s, q, zs, zp, GC_THREADS);
    for (int e = tid; e < q * q; e += GC_THREADS) { const int i = e / q, j = e % q; linvt_out[e] = i <= j ? zs[j * zp + i] : 0.0; }
  }
}

// One CholeskyQR pass, step 2: Z <- Z L^-T in place, 64 rows per CTA, on the FP64 tensor cores (a warp per eight rows), and optionally
// the transposed BF16 splits of the result for the tensor-core projection (the layout of h_splits_kernel).  A triangular solve
// per row, one column after the other, took 15 us for 4096 x 40, 47 us for 16384 x 40 and 186 us for 28672 x 72.
constexpr int OA_ROWS = 64, OA_P = OA_ROWS + 4, OA_OP = OA_ROWS + 1;
__host__ __device__ constexpr size_t oa_smem(int kt) { return sizeof(double) * (size_t)(8 * kt) * (OA_P + 8 * kt + 4) + sizeof(float) * 8 * OA_OP; }
template <int KT>                                       // ceil(q / 8)
__global__ void __launch_bounds__(256)
orth_apply_kernel(float* __restrict__ z, int64_t n_rows, int q, const double* __restrict__ linvt, const int* __restrict__ skip,
                  __nv_bfloat16* __restrict__ hsp, int jp, int64_t ldh) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;
  constexpr int Q8 = 8 * KT, WP = Q8 + 4;
  extern __shared__ __align__(16) double oa_sm[];
  double *As = oa_sm, *Ws = oa_sm + Q8 * OA_P;
  float* Os = reinterpret_cast<float*>(oa_sm);          // [Q8 + 8][OA_OP], over As and Ws once they have been read
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, qq = lane & 3;
  const int64_t p0 = (int64_t)blockIdx.x * OA_ROWS;
#pragma unroll 4
  for (int o = tid; o < OA_ROWS * Q8; o += 256) {
    const int r = o / Q8, i = o % Q8;
    As[i * OA_P + r] = i < q && p0 + r < n_rows ? (double)z[(p0 + r) * q + i] : 0.0;
  }
#pragma unroll 4
  for (int o = tid; o < Q8 * Q8; o += 256) {
    const int i = o / Q8, j = o % Q8;
    Ws[i * WP + j] = i < q && j < q ? linvt[i * q + j] : 0.0;
  }
  __syncthreads();
  double acc[KT][2] = {};
#pragma unroll
  for (int kk = 0; kk < Q8; kk += 4) {
    const double a = As[(kk + qq) * OA_P + 8 * warp + g];
#pragma unroll
    for (int t = kk / 8; t < KT; ++t) metis_small::dmma(acc[t], a, Ws[(kk + qq) * WP + 8 * t + g]);              // L^-T is upper triangular
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < KT; ++t)
#pragma unroll
    for (int e = 0; e < 2; ++e) Os[(8 * t + 2 * qq + e) * OA_OP + 8 * warp + g] = (float)acc[t][e];
  for (int o = tid; o < 8 * OA_OP; o += 256) Os[Q8 * OA_OP + o] = 0.0f;
  __syncthreads();
  for (int o = tid; o < OA_ROWS * q; o += 256) {
    const int r = o / q, j = o - r * q;
    if (p0 + r < n_rows) z[(p0 + r) * q + j] = Os[j * OA_OP + r];
  }
  if (hsp == nullptr) return;
  for (int o = tid; o < jp * (OA_ROWS / 2); o += 256) { // rows beyond n_rows and vectors beyond q are zeros
    const int j = o / (OA_ROWS / 2), r = o % (OA_ROWS / 2) * 2;
    float x = Os[j * OA_OP + r], y = Os[j * OA_OP + r + 1];
    uint32_t w[3];
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
      w[t] = *reinterpret_cast<const uint32_t*>(&h);
      x -= __uint_as_float(w[t] << 16); y -= __uint_as_float(w[t] & 0xFFFF0000u);
      *reinterpret_cast<uint32_t*>(hsp + ((int64_t)t * jp + j) * ldh + p0 + r) = w[t];
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Projection partials: Mp[part][j][col] = sum over the part's sampled rows r of H[r][j] * x[idx[r], col]
// (q x cols per part, row j contiguous).  Thread: two adjacent columns, every second sketch column.
constexpr int PJ_COLS = 256, PJ_ROWS = 32;
template <int NJ4>                                                  // float4 groups of sketch columns per thread
__global__ void __launch_bounds__(256)
project_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, const int* __restrict__ idx, int n_s, int q,
               const float* __restrict__ h, int rows_per_part, float* __restrict__ mp) {
  metis_pdl_wait_trigger();
  __shared__ __align__(16) float hs[2][PJ_ROWS][MAXQ / 2];
  __shared__ int ids[PJ_ROWS];
  const int tid = threadIdx.x, c2 = tid & 127, jg = tid >> 7;       // jg: sketch columns 2*j + jg
  const int64_t col = (int64_t)blockIdx.x * PJ_COLS + c2 * 2;
  const int r_begin = blockIdx.y * rows_per_part, r_end = min(n_s, r_begin + rows_per_part);
  float acc0[NJ4 * 4], acc1[NJ4 * 4];
#pragma unroll
  for (int j = 0; j < NJ4 * 4; ++j) { acc0[j] = 0.0f; acc1[j] = 0.0f; }
  for (int r0 = r_begin; r0 < r_end; r0 += PJ_ROWS) {
    for (int i = tid; i < PJ_ROWS * MAXQ; i += 256) {
      const int rr = i / MAXQ, jj = i % MAXQ;
      hs[jj & 1][rr][jj >> 1] = (r0 + rr < r_end && jj < q) ? h[(int64_t)(r0 + rr) * q + jj] : 0.0f;
    }
    if (tid < PJ_ROWS) ids[tid] = (r0 + tid < r_end) ? idx[r0 + tid] : 0;
    __syncthreads();
    const int nr = min(PJ_ROWS, r_end - r0);
    // the tile's x values first, all loads in flight (inside the loop below each was an L2 round trip per row)
    uint32_t xw[PJ_ROWS];
#pragma unroll
    for (int rr = 0; rr < PJ_ROWS; ++rr) {
      xw[rr] = 0u;
      if (rr < nr) {
        if (col + 1 < cols) xw[rr] = *reinterpret_cast<const uint32_t*>(x + (int64_t)ids[rr] * cols + col);
        else if (col < cols) xw[rr] = (uint32_t)__bfloat16_as_ushort(x[(int64_t)ids[rr] * cols + col]);
      }
    }
#pragma unroll
    for (int rr = 0; rr < PJ_ROWS; ++rr) {
      if (rr >= nr) break;
      const float x0 = __uint_as_float(xw[rr] << 16), x1 = __uint_as_float(xw[rr] & 0xFFFF0000u);
#pragma unroll
      for (int j4 = 0; j4 < NJ4; ++j4) {
        const float4 hv = *reinterpret_cast<const float4*>(&hs[jg][rr][j4 * 4]);
        acc0[j4 * 4 + 0] = fmaf(hv.x, x0, acc0[j4 * 4 + 0]); acc1[j4 * 4 + 0] = fmaf(hv.x, x1, acc1[j4 * 4 + 0]);
        acc0[j4 * 4 + 1] = fmaf(hv.y, x0, acc0[j4 * 4 + 1]); acc1[j4 * 4 + 1] = fmaf(hv.y, x1, acc1[j4 * 4 + 1]);
        acc0[j4 * 4 + 2] = fmaf(hv.z, x0, acc0[j4 * 4 + 2]); acc1[j4 * 4 + 2] = fmaf(hv.z, x1, acc1[j4 * 4 + 2]);
        acc0[j4 * 4 + 3] = fmaf(hv.w, x0, acc0[j4 * 4 + 3]); acc1[j4 * 4 + 3] = fmaf(hv.w, x1, acc1[j4 * 4 + 3]);
      }
    }
    __syncthreads();
  }
  float* dst = mp + (int64_t)blockIdx.y * q * cols;
#pragma unroll
  for (int j = 0; j < NJ4 * 4; ++j)
    if (2 * j + jg < q) {
      if (col < cols) dst[(int64_t)(2 * j + jg) * cols + col] = acc0[j];
      if (col + 1 < cols) dst[(int64_t)(2 * j + jg) * cols + col + 1] = acc1[j];
    }
}

// ------------------------------------------------------------------------------------------------
// Tensor-core helpers (warp-level mma.sync m16n8k16, BF16 operands, FP32 accumulate).  FP32 operands
// are fed as three BF16 terms (hi + lo + lo2 = 24 mantissa bits) so the products stay FP32-accurate.
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}
// three-term BF16 split of a pair of floats: v = hi + lo + lo2 (each term BF16, packed as pairs)
__device__ __forceinline__ void split3(float x, float y, uint32_t& hi, uint32_t& lo, uint32_t& lo2) {
  const __nv_bfloat16 xh = __float2bfloat16_rn(x), yh = __float2bfloat16_rn(y);
  const float xr = x - __bfloat162float(xh), yr = y - __bfloat162float(yh);
  const __nv_bfloat16 xl = __float2bfloat16_rn(xr), yl = __float2bfloat16_rn(yr);
  const float xr2 = xr - __bfloat162float(xl), yr2 = yr - __bfloat162float(yl);
  hi = (uint32_t)__bfloat16_as_ushort(xh) | ((uint32_t)__bfloat16_as_ushort(yh) << 16);
  lo = (uint32_t)__bfloat16_as_ushort(xl) | ((uint32_t)__bfloat16_as_ushort(yl) << 16);
  lo2 = pack_bf16(xr2, yr2);
}

// BF16 splits of the right basis:
//   bs[t][j][col]  (col contiguous; B operand of C = x B, contraction over col); with more than 64 vectors the
//                  layout is by groups of 64 vectors, bs[group][t][j in group][col], so that the three terms of a
//                  group are one contiguous matrix (one launch of the coefficient kernel per group)
//   b6[col][kx]    (optional) per column the six K blocks [Bh | Bl | Bh | Bl2 | Bh | Bl] of the residual product
__global__ void __launch_bounds__(128)
basis_splits_kernel(const float* __restrict__ basis, int64_t cols, int k, int kp, __nv_bfloat16* __restrict__ bs,
                    __nv_bfloat16* __restrict__ b6, int kx) {
  metis_pdl_wait_trigger();
  const int64_t col = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (col >= cols) return;
  if (b6 != nullptr && blockIdx.y == 0)
    for (int z = 6 * kp; z < kx; z += 8) *reinterpret_cast<uint4*>(b6 + col * kx + z) = make_uint4(0u, 0u, 0u, 0u);
  {
    const int j0 = blockIdx.y * 8;                        // grid.y = kp / 8: one group of eight vectors per thread
    uint32_t w[3][4];
#pragma unroll
    for (int jj = 0; jj < 8; jj += 2) {
      const float v0 = j0 + jj < k ? basis[(int64_t)(j0 + jj) * cols + col] : 0.0f;
      const float v1 = j0 + jj + 1 < k ? basis[(int64_t)(j0 + jj + 1) * cols + col] : 0.0f;
      split3(v0, v1, w[0][jj >> 1], w[1][jj >> 1], w[2][jj >> 1]);
    }
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const int grp = j0 / 64, gw = min(64, kp - 64 * grp);
      const int64_t row0 = (int64_t)3 * 64 * grp + (int64_t)t * gw + (j0 - 64 * grp);
#pragma unroll
      for (int jj = 0; jj < 8; ++jj)
        bs[(row0 + jj) * cols + col] = __ushort_as_bfloat16((unsigned short)((w[t][jj >> 1] >> (16 * (jj & 1))) & 0xFFFFu));
    }
    if (b6 != nullptr) {
      const int sel[6] = {0, 1, 0, 2, 0, 1};
#pragma unroll
      for (int term = 0; term < 6; ++term)
        *reinterpret_cast<uint4*>(b6 + col * kx + term * kp + j0) = make_uint4(w[sel[term]][0], w[sel[term]][1], w[sel[term]][2], w[sel[term]][3]);
    }
  }
}

// out[e] = sum over all partials p of in[p][e].  A CTA of four warps owns 32 elements; warp s adds every fourth
// partial (eight loads in flight), the four sums are added in a fixed order: the result does not depend on timing.
__global__ void __launch_bounds__(128)
reduce_gram_kernel(const double* __restrict__ in, int n_in, int nn, double* __restrict__ out,
                   const int* __restrict__ skip) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;
  __shared__ double part[4][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  double a = 0.0;
  if (e < nn) {
    int p = sl;
    for (; p + 28 < n_in; p += 32) {
      double v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = in[(int64_t)(p + 4 * u) * nn + e];
#pragma unroll
      for (int u = 0; u < 8; ++u) a += v[u];
    }
    for (; p < n_in; p += 4) a += in[(int64_t)p * nn + e];
  }
  part[sl][lane] = a;
  __syncthreads();
  if (sl == 0 && e < nn) out[e] = ((part[0][lane] + part[1][lane]) + part[2][lane]) + part[3][lane];
}

// Sums the column slices of the tensor-core broadcast pass in a fixed order: coef[r][j] = sum_s part[s][r][j],
// and writes the FP64 Gram partial of the CTA's 32 rows of C (for Rayleigh-Ritz).
template <int KP>
__global__ void __launch_bounds__(256)
coef_finish_kernel(const float* __restrict__ part, int slices, int64_t rows, float* __restrict__ coef,
                   double* __restrict__ gram_part, __nv_bfloat16* __restrict__ a6, int kx) {
  metis_pdl_wait_trigger();
  __shared__ float cfin[32 * KP];
  const int tid = threadIdx.x;
  const int64_t row0 = (int64_t)blockIdx.x * 32;
  for (int o = tid; o < 32 * KP; o += 256) {
    const int64_t r = row0 + o / KP;
    float v = 0.0f;
    if (r < rows) {
      float t[8];                                          // at most eight slices; all loads in flight, fixed order of the sum
#pragma unroll
      for (int s = 0; s < 8; ++s) t[s] = s < slices ? part[((int64_t)s * rows + r) * KP + (o % KP)] : 0.0f;
#pragma unroll
      for (int s = 0; s < 8; ++s) v += t[s];
      coef[r * KP + (o % KP)] = v;
    }
    cfin[o] = v;
  }
  __syncthreads();
  if (a6 != nullptr) {
    // a6: [rows][kx], per row the six K blocks [Ch | Ch | Cl | Ch | Cl2 | Cl] of the residual product (zero padded)
    for (int o = tid; o < 32 * (KP / 8); o += 256) {
      const int rr = o / (KP / 8), j0 = (o % (KP / 8)) * 8;
      const int64_t r = row0 + rr;
      if (r >= rows) continue;
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = cfin[rr * KP + j0 + e];
      uint4 h, l, l2;
      metis_split3x8(v, h, l, l2);
      __nv_bfloat16* dst = a6 + r * kx + j0;
      *reinterpret_cast<uint4*>(dst) = h; *reinterpret_cast<uint4*>(dst + KP) = h; *reinterpret_cast<uint4*>(dst + 2 * KP) = l;
      *reinterpret_cast<uint4*>(dst + 3 * KP) = h; *reinterpret_cast<uint4*>(dst + 4 * KP) = l2; *reinterpret_cast<uint4*>(dst + 5 * KP) = l;
      if (j0 == 0)
        for (int z = 6 * KP; z < kx; z += 8) *reinterpret_cast<uint4*>(a6 + r * kx + z) = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (gram_part) {
    __shared__ double cd[32 * KP];                      // converted once: FP32 -> FP64 is a slow-rate instruction
    for (int o = tid; o < 32 * KP; o += 256) cd[o] = (double)cfin[o];
    __syncthreads();
    for (int o = tid; o < KP * KP; o += 256) {
      const int i = o / KP, j = o % KP;
      double a = 0.0;
#pragma unroll 8
      for (int r = 0; r < 32; ++r) a += cd[r * KP + i] * cd[r * KP + j];
      gram_part[(int64_t)blockIdx.x * KP * KP + o] = a;
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Sketch of gathered rows (mma.sync): Zp[chunk][row][j] = sum over the chunk's columns of x[idx[row], col] * Omega[col, j].
// One CTA = 256 sampled rows x one column chunk (`ccols` = 64 or 256 columns, see sketch_chunk_cols); Omega's slice
// is generated once per CTA (Philox + quantile table) straight into shared memory, transposed to [j][col] BF16 (its
// values are BF16 by construction, so the products are exact and only the FP32 accumulation rounds).  Optionally also
// reduces amax|x| over the rows it reads.  A full sketch of an aligned operand does not come here: it runs on the
// tcgen05 kernel of the broadcast pass (omega_rows_kernel + metis_launch_coeff_tc in its raw mode).
constexpr int SKM_ROWS = 256, SKM_COLS = 256, SKM_PITCH = SKM_COLS + 8;
template <int NT>                                      // sketch columns / 8, rounded up
__global__ void __launch_bounds__(256)
sketch_mma_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, const int* __restrict__ idx, int n_s, int q,
                  uint64_t seed, const __nv_bfloat16* __restrict__ lut, float* __restrict__ zp, float* __restrict__ amax_out,
                  int ccols) {
  metis_pdl_wait_trigger();
  extern __shared__ __align__(16) unsigned char smem[];
  __nv_bfloat16* om = reinterpret_cast<__nv_bfloat16*>(smem);          // [NT*8][SKM_PITCH]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int64_t col0 = (int64_t)blockIdx.y * ccols;        // ccols <= SKM_COLS columns per CTA
  const int row0 = blockIdx.x * SKM_ROWS + warp * 32;
  const int ncols = (int)min((int64_t)ccols, cols - col0);
  for (int i = tid; i < NT * 8 * SKM_PITCH; i += 256) om[i] = __float2bfloat16_rn(0.0f);
  __syncthreads();
  const uint64_t e_lo = (uint64_t)col0 * q, e_hi = (uint64_t)(col0 + ncols) * q;
  for (uint64_t blk = (e_lo >> 3) + tid; blk <= ((e_hi - 1) >> 3); blk += 256) {
    const uint4 w = metis_philox_block(blk, seed, METIS_STREAM_OMEGA);
#pragma unroll
    for (uint32_t h = 0; h < 8; ++h) {
      const uint64_t e = (blk << 3) + h;
      if (e >= e_lo && e < e_hi) {
        const uint32_t rel = (uint32_t)(e - e_lo);
        om[(rel % q) * SKM_PITCH + rel / q] = lut[metis_u16_of(w, h)];
      }
    }
  }
  __syncthreads();
  float acc[2][NT][4];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.0f;
  const bool v0 = row0 + g < n_s, v1 = row0 + g + 8 < n_s, v2 = row0 + g + 16 < n_s, v3 = row0 + g + 24 < n_s;
  const __nv_bfloat16* p0 = x + (int64_t)(v0 ? idx[row0 + g] : 0) * cols + col0;
  const __nv_bfloat16* p1 = x + (int64_t)(v1 ? idx[row0 + g + 8] : 0) * cols + col0;
  const __nv_bfloat16* p2 = x + (int64_t)(v2 ? idx[row0 + g + 16] : 0) * cols + col0;
  const __nv_bfloat16* p3 = x + (int64_t)(v3 ? idx[row0 + g + 24] : 0) * cols + col0;
  uint32_t amax2 = 0u;
#pragma unroll 2
  for (int ks = 0; ks < ncols / 16; ++ks) {
    const int kk = ks * 16 + 2 * t;
    uint32_t a[2][4];
    a[0][0] = v0 ? *reinterpret_cast<const uint32_t*>(p0 + kk) : 0u;
    a[0][1] = v1 ? *reinterpret_cast<const uint32_t*>(p1 + kk) : 0u;
    a[0][2] = v0 ? *reinterpret_cast<const uint32_t*>(p0 + kk + 8) : 0u;
    a[0][3] = v1 ? *reinterpret_cast<const uint32_t*>(p1 + kk + 8) : 0u;
    a[1][0] = v2 ? *reinterpret_cast<const uint32_t*>(p2 + kk) : 0u;
    a[1][1] = v3 ? *reinterpret_cast<const uint32_t*>(p3 + kk) : 0u;
    a[1][2] = v2 ? *reinterpret_cast<const uint32_t*>(p2 + kk + 8) : 0u;
    a[1][3] = v3 ? *reinterpret_cast<const uint32_t*>(p3 + kk + 8) : 0u;
    if (amax_out) {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t ab = a[m][e] & 0x7FFF7FFFu;
          amax2 = max(ab & 0xFFFFu, amax2 & 0xFFFFu) | (max(ab >> 16, amax2 >> 16) << 16);
        }
    }
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const __nv_bfloat16* bp = om + (n * 8 + g) * SKM_PITCH + kk;
      const uint32_t b0 = *reinterpret_cast<const uint32_t*>(bp), b1 = *reinterpret_cast<const uint32_t*>(bp + 8);
      mma_bf16(acc[0][n], a[0], b0, b1);
      mma_bf16(acc[1][n], a[1], b0, b1);
    }
  }
  float* dst = zp + (int64_t)blockIdx.y * n_s * q;
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n) {
      const int r = row0 + m * 16 + g, j = n * 8 + 2 * t;
      if (r < n_s) { if (j < q) dst[(int64_t)r * q + j] = acc[m][n][0]; if (j + 1 < q) dst[(int64_t)r * q + j + 1] = acc[m][n][1]; }
      if (r + 8 < n_s) { if (j < q) dst[(int64_t)(r + 8) * q + j] = acc[m][n][2]; if (j + 1 < q) dst[(int64_t)(r + 8) * q + j + 1] = acc[m][n][3]; }
    }
  if (amax_out) {
    uint32_t am = max((amax2 & 0xFFFFu) << 16, amax2 & 0xFFFF0000u);      // ordered bit patterns: a NaN survives
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) am = max(am, __shfl_xor_sync(0xFFFFFFFFu, am, o));
    if (lane == 0) atomicMax(reinterpret_cast<unsigned int*>(amax_out), am);
  }
}

// Full-mode sketch on the tcgen05 path: Omega is written once, transposed and zero-padded to nb rows
// (omt[j][col], BF16: its values are BF16 by construction), and Z = X Omega runs on the same kernel as the
// coefficient pass.  One thread per Philox block of eight consecutive elements e = col * q + j.
__global__ void __launch_bounds__(256)
omega_rows_kernel(int64_t cols, int q, int nb, uint64_t seed, const __nv_bfloat16* __restrict__ lut, __nv_bfloat16* __restrict__ omt) {
  metis_pdl_wait_trigger();
  const uint64_t total = (uint64_t)cols * (uint64_t)q;
  const uint64_t blk = (uint64_t)blockIdx.x * 256 + threadIdx.x;
  if (blk < (total + 7) / 8) {
    const uint4 w = metis_philox_block(blk, seed, METIS_STREAM_OMEGA);
#pragma unroll
    for (uint32_t h = 0; h < 8; ++h) {
      const uint64_t e = (blk << 3) + h;
      if (e < total) omt[(e % q) * cols + e / q] = lut[metis_u16_of(w, h)];
    }
  }
  // rows q .. nb-1 are zero
  const int64_t pad = (int64_t)(nb - q) * cols;
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < pad; i += (int64_t)gridDim.x * 256)
    omt[(int64_t)q * cols + i] = __float2bfloat16_rn(0.0f);
}

// m[j][col] = sum over slices s of part[s][col][j], j < q (the tensor-core projection writes M transposed, jp wide)
__global__ void __launch_bounds__(256)
reduce_proj_kernel(const float* __restrict__ part, int slices, int64_t cols, int jp, int q, float* __restrict__ m) {
  metis_pdl_wait_trigger();
  __shared__ float t[32][33];
  const int64_t c0 = (int64_t)blockIdx.x * 32;
  const int j0 = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int r = ty; r < 32; r += 8) {                     // r: column of x inside the tile, tx: sketch index
    float acc = 0.0f;
    if (c0 + r < cols && j0 + tx < q) {
      float v[8];                                           // at most eight slices
#pragma unroll
      for (int s = 0; s < 8; ++s) v[s] = s < slices ? part[((int64_t)s * cols + c0 + r) * jp + j0 + tx] : 0.0f;
#pragma unroll
      for (int s = 0; s < 8; ++s) acc += v[s];
    }
    t[r][tx] = acc;
  }
  __syncthreads();
  for (int r = ty; r < 32; r += 8)                        // r: sketch index, tx: column
    if (j0 + r < q && c0 + tx < cols) m[(int64_t)(j0 + r) * cols + c0 + tx] = t[tx][r];
}

// z[r * ldz + j] = sum over slices s of part[s][r][j], j < q (part rows are nb wide); fixed order
__global__ void __launch_bounds__(256)
reduce_sketch_kernel(const float* __restrict__ part, int slices, int64_t rows, int nb, int q, float* __restrict__ z, int ldz) {
  metis_pdl_wait_trigger();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= rows * q) return;
  const int64_t r = i / q;
  const int j = (int)(i % q);
  float t[8], acc = 0.0f;                                 // at most eight slices
#pragma unroll
  for (int s = 0; s < 8; ++s) t[s] = s < slices ? part[((int64_t)s * rows + r) * nb + j] : 0.0f;
#pragma unroll
  for (int s = 0; s < 8; ++s) acc += t[s];
  z[r * ldz + j] = acc;
}

// Tensor-core projection: Mp[part][j][col] = sum over the part's sampled rows r of H[r][j] * x[idx[r], col].
// The contraction runs over rows of the row-major x, so x tiles are staged in shared memory and read back
// transposed with ldmatrix; H (FP32) is fed as three BF16 terms.  CTA = 128 columns x one slab of rows.
// ------------------------------------------------------------------------------------------------
// Projection M = H^T x over many rows (every row in FULL mode), software-pipelined: the CTA owns 128 columns and
// a slab of rows, and walks the slab in chunks of 64 rows through a three-stage cp.async ring (x rows gathered
// by idx, the three BF16 terms of H pre-split and transposed by h_splits_kernel), so the loads of chunk c + 2
// overlap the MMAs of chunk c.  Same partial layout as project_kernel: Mp[part][j][col].
constexpr int PP_COLS = 128, PP_K = 64, PP_STAGES = 3, PP_XP = PP_COLS + 8, PP_HP = PP_K + 8;

// hsp[sp][j][r] (r contiguous, ldh >= rows rounded up to 64, zero padded): three-term BF16 split of H[r][j]
__global__ void __launch_bounds__(256)
h_splits_kernel(const float* __restrict__ h, int n_s, int q, int jp, int ldh, __nv_bfloat16* __restrict__ hsp, int pitch_h) {
  metis_pdl_wait_trigger();
  const int r = blockIdx.x * 256 + threadIdx.x, j = blockIdx.y;
  if (r >= ldh) return;
  const float v = (r < n_s && j < q) ? h[(int64_t)r * pitch_h + j] : 0.0f;
  const __nv_bfloat16 hh = __float2bfloat16_rn(v);
  const float r1 = v - __bfloat162float(hh);
  const __nv_bfloat16 hl = __float2bfloat16_rn(r1);
  hsp[((int64_t)0 * jp + j) * ldh + r] = hh;
  hsp[((int64_t)1 * jp + j) * ldh + r] = hl;
  hsp[((int64_t)2 * jp + j) * ldh + r] = __float2bfloat16_rn(r1 - __bfloat162float(hl));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int bytes = valid ? 16 : 0;                      // 0: the 16 destination bytes are zero-filled
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

template <int MT>                                      // sketch columns / 16, rounded up
__global__ void __launch_bounds__(256)
project_pipe_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, const int* __restrict__ idx, int n_s, int q,
                    const __nv_bfloat16* __restrict__ hsp, int ldh, int rows_per_part, float* __restrict__ mp) {
  metis_pdl_wait_trigger();
  extern __shared__ __align__(16) unsigned char psm[];
  constexpr int XS_BYTES = PP_K * PP_XP * 2, HS_BYTES = 3 * MT * 16 * PP_HP * 2, STAGE = XS_BYTES + HS_BYTES;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(psm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int64_t col0 = (int64_t)blockIdx.x * PP_COLS;
  const int r_begin = blockIdx.y * rows_per_part, r_end = min(n_s, r_begin + rows_per_part);
  const int n_chunks = (r_end - r_begin + PP_K - 1) / PP_K;
  float acc[MT][2][4];
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.0f;

  auto load_chunk = [&](int c) {
    const int st = c % PP_STAGES;
    const int r0 = r_begin + c * PP_K;
    const uint32_t xs = sbase + (uint32_t)st * STAGE, hs = xs + XS_BYTES;
    for (int i = tid; i < PP_K * (PP_COLS / 8); i += 256) {
      const int rr = i >> 4, c8 = (i & 15) * 8;
      const bool ok = r0 + rr < r_end && col0 + c8 + 8 <= cols;
      const __nv_bfloat16* src = ok ? x + (int64_t)idx[r0 + rr] * cols + col0 + c8 : x;
      cp_async16(xs + (uint32_t)(rr * PP_XP + c8) * 2u, src, ok);
    }
    for (int i = tid; i < 3 * MT * 16 * (PP_K / 8); i += 256) {
      const int row = i >> 3, k8 = (i & 7) * 8;          // row = sp * MT*16 + j
      cp_async16(hs + (uint32_t)(row * PP_HP + k8) * 2u, hsp + (int64_t)row * ldh + r0 + k8, true);
    }
  };

  for (int c = 0; c < PP_STAGES - 1; ++c) {
    if (c < n_chunks) load_chunk(c);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int c = 0; c < n_chunks; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(PP_STAGES - 2) : "memory");
    __syncthreads();                                     // chunk c has landed; everyone is done with chunk c - 1
    if (c + PP_STAGES - 1 < n_chunks) load_chunk(c + PP_STAGES - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int st = c % PP_STAGES;
    const uint32_t xs = sbase + (uint32_t)st * STAGE, hs = xs + XS_BYTES;
#pragma unroll
    for (int ks = 0; ks < PP_K / 16; ++ks) {
      uint32_t b[2][2];
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const uint32_t addr = xs + (uint32_t)((ks * 16 + (lane & 15)) * PP_XP + (warp * 2 + n) * 8) * 2u;
        asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(b[n][0]), "=r"(b[n][1]) : "r"(addr));
      }
#pragma unroll
      for (int sp = 0; sp < 3; ++sp)
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          uint32_t a[4];
          const uint32_t addr = hs + (uint32_t)(((sp * MT + m) * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * PP_HP + ks * 16 + (lane >> 4) * 8) * 2u;
          asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                       : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]) : "r"(addr));
          mma_bf16(acc[m][0], a, b[0][0], b[0][1]);
          mma_bf16(acc[m][1], a, b[1][0], b[1][1]);
        }
    }
  }
  float* dst = mp + (int64_t)blockIdx.y * q * cols;
#pragma unroll
  for (int m = 0; m < MT; ++m)
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int j = m * 16 + g;
      const int64_t col = col0 + (warp * 2 + n) * 8 + 2 * t;
      if (col + 1 < cols) {
        if (j < q) *reinterpret_cast<float2*>(dst + (int64_t)j * cols + col) = make_float2(acc[m][n][0], acc[m][n][1]);
        if (j + 8 < q) *reinterpret_cast<float2*>(dst + (int64_t)(j + 8) * cols + col) = make_float2(acc[m][n][2], acc[m][n][3]);
      }
    }
}


// ------------------------------------------------------------------------------------------------
// Factors from eigenvectors:  out[j][p] = scale_j sum_i src(i, p) W[i][j]  for a tile of 64 positions p (columns or rows of the
// operand) and every j < k, on the FP64 tensor cores; i <= 72, j <= 64.  Used for the right basis (src = M, W = evecs), the left
// factor (src = H or C) and the Rayleigh-Ritz rotation of the basis.  One kernel per stage of the chain does all that is
// derived from the product - BF16 splits, the operands of the residual product, tensor amax, the sign decision - because the chain is
// latency: the right basis, its sign, its splits, the left factor and its splits were six launches (28 us at
// 4096 x 4096, k = 32; now 11 us in two), and beside a persistent residual pass, on the few SMs it leaves, FP32 multiply-adds with 72
// registers of basis values a thread took 775 us for 28672 x 64.
//
// Sign convention: the entry of largest magnitude of a right vector (lowest index on ties) is positive.  The contest is an
// atomic maximum over keys (magnitude bits, inverted column, sign), whatever the order of arrival; the factors stay
// unsigned until the factor quantizer, which reads the key's sign and flips both (the residual C B^T does not see it).
constexpr int FR_POS = 64, FR_P = FR_POS + 4, FR_OP = FR_POS + 1;
__host__ __device__ constexpr size_t fr_smem(int n_in) { return sizeof(double) * 2 * (size_t)((n_in + 7) / 8 * 8 < 40 ? 40 : (n_in + 7) / 8 * 8) * FR_P; }
__device__ __forceinline__ unsigned long long sign_key(float v, int64_t col) {
  const uint32_t b = __float_as_uint(v);
  return ((unsigned long long)(b & 0x7FFFFFFFu) << 32) | ((0x7FFFFFFFull - (unsigned long long)col) << 1) | (v < 0.0f ? 1ull : 0ull);
}

// Os[j][p] = (float)(scale[j] * sum); rows j in [k, 8 KT + 8) are zero.  src(i, p) = src[i * stride_i + p * stride_p], one of the strides 1.
template <int KT>
__device__ __forceinline__ void factor_tile(const float* __restrict__ src, int64_t n_pos, int64_t p0, int64_t stride_i, int64_t stride_p, int n_in,
                                            const double* __restrict__ w, int ldw, int k, const double* scale, double* As, double* Ws, float* Os) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3, n8 = (n_in + 7) & ~7;
  if (stride_p == 1) {
#pragma unroll 4
    for (int o = tid; o < n8 * FR_POS; o += 256) {
      const int i = o / FR_POS, c = o % FR_POS;
      As[i * FR_P + c] = i < n_in && p0 + c < n_pos ? (double)src[i * stride_i + p0 + c] : 0.0;
    }
  } else {
#pragma unroll 4
    for (int o = tid; o < n8 * FR_POS; o += 256) {
      const int c = o / n8, i = o - c * n8;
      As[i * FR_P + c] = i < n_in && p0 + c < n_pos ? (double)src[(p0 + c) * stride_p + i] : 0.0;
    }
  }
#pragma unroll 4
  for (int o = tid; o < n8 * 8 * KT; o += 256) {
    const int i = o / (8 * KT), j = o % (8 * KT);
    Ws[i * FR_P + j] = i < n_in && j < k ? w[i * ldw + j] : 0.0;
  }
  __syncthreads();
  double acc[KT][2] = {};
  for (int kk = 0; kk < n8; kk += 4) {
    const double a = As[(kk + q) * FR_P + 8 * warp + g];
#pragma unroll
    for (int t = 0; t < KT; ++t) metis_small::dmma(acc[t], a, Ws[(kk + q) * FR_P + 8 * t + g]);
  }
  __syncthreads();                                      // Os lies over As
#pragma unroll
  for (int t = 0; t < KT; ++t)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int j = 8 * t + 2 * q + e;
      Os[j * FR_OP + 8 * warp + g] = j < k ? (float)(scale != nullptr ? acc[t][e] * scale[j] : acc[t][e]) : 0.0f;
    }
  for (int o = tid; o < 8 * FR_OP; o += 256) Os[8 * KT * FR_OP + o] = 0.0f;
  __syncthreads();
}

// the tile's entries into the sign contest and the tensor amax, one warp per vector
__device__ __forceinline__ void sign_contest(const float* Os, int k, int64_t p0, int64_t n_pos, unsigned long long* keys, float* amax) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t top = 0u;
  for (int j = warp; j < k; j += 8) {
    unsigned long long key = p0 + lane < n_pos ? sign_key(Os[j * FR_OP + lane], p0 + lane) : 0ull;
    if (p0 + lane + 32 < n_pos) { const unsigned long long o = sign_key(Os[j * FR_OP + lane + 32], p0 + lane + 32); key = o > key ? o : key; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) { const unsigned long long x = __shfl_xor_sync(0xFFFFFFFFu, key, o); key = x > key ? x : key; }
    if (lane == 0) atomicMax(keys + j, key);
    top = max(top, (uint32_t)(key >> 32));
  }
  if (lane == 0 && top != 0u) atomicMax(reinterpret_cast<unsigned int*>(amax), top);
}

// Right basis B[j][col] = sum_i evecs[i][j] M[i][col] / s_j, s_j = sqrt(eval_j), and its BF16 splits (see basis_splits_kernel; bs
// is optional).  keys (FULL mode, where this is the right factor itself): the sign contest.
template <int KT>
__global__ void __launch_bounds__(256)
basis_kernel(const float* __restrict__ m, int64_t cols, int q, int k, int kp, const double* __restrict__ evals, const double* __restrict__ evecs,
             float* __restrict__ basis, __nv_bfloat16* __restrict__ bs, __nv_bfloat16* __restrict__ b6, int kx,
             float* __restrict__ sigma_out, unsigned long long* __restrict__ keys, float* __restrict__ amax_out) {
  metis_pdl_wait_trigger();
  extern __shared__ __align__(16) double fr_sm[];
  __shared__ double scale[FR_POS];
  double *As = fr_sm, *Ws = fr_sm + ((q + 7) / 8 * 8 < 40 ? 40 : (q + 7) / 8 * 8) * FR_P;
  float* Os = reinterpret_cast<float*>(As);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t p0 = (int64_t)blockIdx.x * FR_POS;
  if (tid < k) {
    const double sv = sqrt(fmax(evals[tid], 0.0));
    scale[tid] = sv > 0.0 ? 1.0 / sv : 0.0;
    if (blockIdx.x == 0 && sigma_out != nullptr) sigma_out[tid] = (float)sv;
  }
  factor_tile<KT>(m, cols, p0, cols, 1, q, evecs, q, k, scale, As, Ws, Os);
  for (int o = tid; o < k * FR_POS; o += 256) {
    const int j = o / FR_POS, c = o % FR_POS;
    if (p0 + c < cols) basis[(int64_t)j * cols + p0 + c] = Os[j * FR_OP + c];
  }
  const int64_t col2 = p0 + 2 * lane;                   // a pair of columns (their number is a multiple of 16)
  for (int j = warp; j < kp && bs != nullptr; j += 8) {
    uint32_t h, l, l2;
    split3(Os[j * FR_OP + 2 * lane], Os[j * FR_OP + 2 * lane + 1], h, l, l2);
    if (col2 < cols) {
      *reinterpret_cast<uint32_t*>(bs + (int64_t)j * cols + col2) = h;
      *reinterpret_cast<uint32_t*>(bs + (int64_t)(kp + j) * cols + col2) = l;
      *reinterpret_cast<uint32_t*>(bs + (int64_t)(2 * kp + j) * cols + col2) = l2;
    }
  }
  for (int o = tid; o < FR_POS * (kp / 8); o += 256) {
    const int c = o / (kp / 8), j0 = o % (kp / 8) * 8;  // consecutive threads: consecutive 16-byte groups of a column's row
    const int64_t col = p0 + c;
    if (col >= cols) break;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = Os[(j0 + e) * FR_OP + c];
    uint4 h, l, l2;
    metis_split3x8(v, h, l, l2);
    __nv_bfloat16* dst = b6 + col * kx + j0;
    *reinterpret_cast<uint4*>(dst) = h; *reinterpret_cast<uint4*>(dst + kp) = l; *reinterpret_cast<uint4*>(dst + 2 * kp) = h;
    *reinterpret_cast<uint4*>(dst + 3 * kp) = l2; *reinterpret_cast<uint4*>(dst + 4 * kp) = h; *reinterpret_cast<uint4*>(dst + 5 * kp) = l;
    if (j0 == 0)
      for (int z = 6 * kp; z < kx; z += 8) *reinterpret_cast<uint4*>(b6 + col * kx + z) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (keys != nullptr) sign_contest(Os, k, p0, cols, keys, amax_out);
}

// The factors of a decomposition, unsigned.  Blocks below n_right: right[j][col] = sum_i basis[i][col] W[i][j] and the sign contest;
// the others: left[j][r] = s_j sum_i src[r * ld + i] W[i][j] with s_j = 1 / sqrt(eval_j) when evals is given (Rayleigh-Ritz; sigma_out = sqrt(eval_j)),
// and from it the coefficients left * sigma of the residual product (FULL mode) as its BF16 operand a6.
struct FactorsArgs {
  const double* w; int ldw, n_in, k, kp;
  const float* basis; int64_t cols; float* right; unsigned long long* keys; float* amax_right;
  const float* src; int64_t ld, rows; const double* evals; float* left; float* sigma_out; float* amax_left;
  const float* sigma_for_coef; __nv_bfloat16* a6; int kx;
};
template <int KT>
__global__ void __launch_bounds__(256)
factors_kernel(FactorsArgs f, int n_right) {
  metis_pdl_wait_trigger();
  extern __shared__ __align__(16) double fr_sm[];
  __shared__ double scale[FR_POS];
  double *As = fr_sm, *Ws = fr_sm + ((f.n_in + 7) / 8 * 8 < 40 ? 40 : (f.n_in + 7) / 8 * 8) * FR_P;
  float* Os = reinterpret_cast<float*>(As);
  const int tid = threadIdx.x, k = f.k;
  if ((int)blockIdx.x < n_right) {
    const int64_t p0 = (int64_t)blockIdx.x * FR_POS;
    factor_tile<KT>(f.basis, f.cols, p0, f.cols, 1, f.n_in, f.w, f.ldw, k, nullptr, As, Ws, Os);
    for (int o = tid; o < k * FR_POS; o += 256) {
      const int j = o / FR_POS, c = o % FR_POS;
      if (p0 + c < f.cols) f.right[(int64_t)j * f.cols + p0 + c] = Os[j * FR_OP + c];
    }
    sign_contest(Os, k, p0, f.cols, f.keys, f.amax_right);
    return;
  }
  const int64_t p0 = (int64_t)((int)blockIdx.x - n_right) * FR_POS;
  if (f.evals != nullptr && tid < k) {
    const double lam = sqrt(fmax(f.evals[tid], 0.0));
    scale[tid] = lam > 0.0 ? 1.0 / lam : 0.0;
    if ((int)blockIdx.x == n_right) f.sigma_out[tid] = (float)lam;
  }
  factor_tile<KT>(f.src, f.rows, p0, 1, f.ld, f.n_in, f.w, f.ldw, k, f.evals != nullptr ? scale : nullptr, As, Ws, Os);
  float am = 0.0f;
  for (int o = tid; o < k * FR_POS; o += 256) {
    const int j = o / FR_POS, c = o % FR_POS;
    const float v = Os[j * FR_OP + c];
    if (p0 + c < f.rows) { f.left[(int64_t)j * f.rows + p0 + c] = v; am = fmaxf(am, fabsf(v)); }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) am = fmaxf(am, __shfl_xor_sync(0xFFFFFFFFu, am, o));
  if ((tid & 31) == 0) atomicMax(reinterpret_cast<unsigned int*>(f.amax_left), __float_as_uint(am));
  if (f.sigma_for_coef == nullptr) return;
  const int kp = f.kp;
  for (int o = tid; o < FR_POS * (kp / 8); o += 256) {
    const int c = o / (kp / 8), j0 = o % (kp / 8) * 8;
    const int64_t r = p0 + c;
    if (r >= f.rows) break;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = j0 + e < k ? Os[(j0 + e) * FR_OP + c] * f.sigma_for_coef[j0 + e] : 0.0f;
    uint4 h, l, l2;
    metis_split3x8(v, h, l, l2);
    __nv_bfloat16* dst = f.a6 + r * f.kx + j0;
    *reinterpret_cast<uint4*>(dst) = h; *reinterpret_cast<uint4*>(dst + kp) = h; *reinterpret_cast<uint4*>(dst + 2 * kp) = l;
    *reinterpret_cast<uint4*>(dst + 3 * kp) = h; *reinterpret_cast<uint4*>(dst + 4 * kp) = l2; *reinterpret_cast<uint4*>(dst + 5 * kp) = l;
    if (j0 == 0)
      for (int z = 6 * kp; z < f.kx; z += 8) *reinterpret_cast<uint4*>(f.a6 + r * f.kx + z) = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Columns per sketch CTA: a sampled sketch has few rows, so narrow chunks are what gives it enough CTAs; a full
// sketch has one CTA per 256 rows already and wide chunks keep the partial buffer small.
// accumulator columns of the tensor-core sketch: k + p rounded up to what the coefficient kernel is built for
int sketch_tc_cols(int q) { return q <= 48 ? 48 : 96; }

int sketch_chunk_cols(int64_t n_s) { return n_s <= 512 ? 64 : SKM_COLS; }

struct SplitWs {
  size_t amax, idx, zp, omt, z, gram, gram1, linv, evals, evecs, mp, m, basis, coef, keys, evals2, evecs2, bs,
      gram_c, part, a6, b6, hsp, total;
};

constexpr int PJ_MAX_PARTS = 16;

int project_parts(int64_t n_s, int64_t cols, int* rows_per_part) {
  const int64_t col_chunks = metis_ceil_div(cols, PJ_COLS);
  int64_t parts = metis_ceil_div(2 * 148, col_chunks);          // aim at two CTAs per SM
  if (parts > PJ_MAX_PARTS) parts = PJ_MAX_PARTS;
  if (parts > metis_ceil_div(n_s, 16)) parts = metis_ceil_div(n_s, 16);
  if (parts < 1) parts = 1;
  int64_t rpp = metis_ceil_div(n_s, parts);
  rpp = metis_ceil_div(rpp, 16) * 16;
  *rows_per_part = (int)rpp;
  return (int)metis_ceil_div(n_s, rpp);
}

SplitWs split_ws_layout(int64_t rows, int64_t cols, int k, int p, int64_t n_s) {
  SplitWs w{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const int q = k + p;
  const int64_t chunks = metis_ceil_div(cols, sketch_chunk_cols(n_s));
  w.amax = take(256);
  w.idx = take(sizeof(int) * (size_t)n_s);
  // the full-mode tensor-core sketch writes slices x rows x nb partials into the same buffer
  const int nb_sk = sketch_tc_cols(q);
  const size_t zp_mma = (size_t)chunks * n_s * q, zp_tc = (size_t)metis_coeff_slices(rows, cols, nullptr) * rows * nb_sk;
  w.zp = take(sizeof(float) * (zp_mma > zp_tc ? zp_mma : zp_tc));
  w.omt = take(sizeof(__nv_bfloat16) * (size_t)nb_sk * cols);
  w.z = take(sizeof(float) * (size_t)n_s * q);
  w.gram = take(sizeof(double) * 64 * MAXQ * MAXQ);
  w.linv = take(sizeof(double) * (MAXQ * MAXQ + MAXQ));
  w.gram1 = take(sizeof(double) * MAXQ * MAXQ);
  w.evals = take(sizeof(double) * MAXQ);
  w.evecs = take(sizeof(double) * MAXQ * MAXQ);
  {
    const size_t per_col_mma = (size_t)PJ_MAX_PARTS * q, per_col_tc = (size_t)8 * ((q + 15) / 16 * 16);   // tensor-core projection: <= 8 slices x jp
    w.mp = take(sizeof(float) * (per_col_mma > per_col_tc ? per_col_mma : per_col_tc) * cols);
  }
  w.m = take(sizeof(float) * (size_t)q * cols);
  w.basis = take(sizeof(float) * (size_t)k * cols);
  const int kp = (k + 15) / 16 * 16;
  w.coef = take(sizeof(float) * (size_t)kp * rows);
  w.part = take(sizeof(float) * (size_t)metis_coeff_slices(rows, cols, nullptr) * kp * rows);
  w.a6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * rows);
  w.b6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * cols);
  w.hsp = take(n_s >= 1024 ? sizeof(__nv_bfloat16) * 3 * (size_t)((q + 15) / 16 * 16) * (size_t)((n_s + 63) / 64 * 64) : 0);
  w.bs = take(sizeof(__nv_bfloat16) * 3 * (size_t)kp * cols);
  w.gram_c = take(sizeof(double) * (size_t)metis_ceil_div(rows, 32) * kp * kp);
  w.keys = take(sizeof(unsigned long long) * MAXQ);
  w.evals2 = take(sizeof(double) * MAXQ);
  w.evecs2 = take(sizeof(double) * MAXQ * MAXQ);
  w.total = off;
  return w;
}

int gram_parts(int64_t n_rows, int64_t* rows_per_part) {
  int parts = (int)metis_ceil_div(n_rows, 64);
  if (parts > 64) parts = 64;
  if (parts < 1) parts = 1;
  int64_t rpp = metis_ceil_div(n_rows, parts);
  rpp = metis_ceil_div(rpp, GR_TILE) * GR_TILE;
  *rows_per_part = rpp;
  return (int)metis_ceil_div(n_rows, rpp);
}

metis_status_t launch_eig(cudaStream_t s, const double* g, int n, int ld, double* evals, double* evecs) {
  const size_t smem = metis_small::eig_smem(n);
#define METIS_EIG(NT8) case NT8: METIS_CUDA_TRY(metis_launch_pdl((metis_small::eig_kernel<NT8>), dim3(1), dim3(metis_small::eig_threads(NT8)), smem, s, g, n, ld, evals, evecs)); break
  switch ((n + 7) / 8) {
    METIS_EIG(1); METIS_EIG(2); METIS_EIG(3); METIS_EIG(4); METIS_EIG(5); METIS_EIG(6); METIS_EIG(7); METIS_EIG(8); METIS_EIG(9);
    default: return METIS_ERR_SHAPE;
  }
#undef METIS_EIG
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

template <int NJ4>
void launch_project(dim3 grid, cudaStream_t s, const __nv_bfloat16* x, int64_t cols, const int* idx, int n_s, int q,
                    const float* h, int rpp, float* mp) {
  (void)(metis_launch_pdl((project_kernel<NJ4>), dim3(grid), dim3(256), (size_t)(0), s, x, cols, idx, n_s, q, h, rpp, mp)); METIS_COUNT_LAUNCH();
}

metis_status_t launch_orth_apply(cudaStream_t s, float* z, int64_t n_s, int q, const double* linvt, const int* skip, __nv_bfloat16* hsp, int jp, int64_t ldh) {
  const dim3 grid((unsigned)metis_ceil_div(n_s, OA_ROWS));
#define METIS_OA(KT) METIS_CUDA_TRY(metis_launch_pdl((orth_apply_kernel<KT>), grid, dim3(256), oa_smem(KT), s, z, n_s, q, linvt, skip, hsp, jp, ldh)); break
  switch ((q + 7) / 8) {
    case 1: METIS_OA(1); case 2: METIS_OA(2); case 3: METIS_OA(3); case 4: METIS_OA(4); case 5: METIS_OA(5); case 6: METIS_OA(6); case 7: METIS_OA(7); case 8: METIS_OA(8);
    default: METIS_OA(9);
  }
#undef METIS_OA
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}
template <int KT>
metis_status_t launch_basis_kt(cudaStream_t s, int ctas, size_t smem, const float* m, int64_t cols, int q, int k, int kp, const double* evals, const double* evecs, float* basis,
                               __nv_bfloat16* bs, __nv_bfloat16* b6, int kx, float* sigma_out, unsigned long long* keys, float* amax_out) {
  METIS_CUDA_TRY(metis_launch_pdl((basis_kernel<KT>), dim3((unsigned)ctas), dim3(256), smem, s, m, cols, q, k, kp, evals, evecs, basis, bs, b6, kx, sigma_out, keys, amax_out));
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}
template <typename... A>
metis_status_t launch_basis(cudaStream_t s, int ctas, size_t smem, const float* m, int64_t cols, int q, int k, A... rest) {
  switch ((k + 7) / 8) {
    case 1: return launch_basis_kt<1>(s, ctas, smem, m, cols, q, k, rest...);
    case 2: return launch_basis_kt<2>(s, ctas, smem, m, cols, q, k, rest...);
    case 3: return launch_basis_kt<3>(s, ctas, smem, m, cols, q, k, rest...);
    case 4: return launch_basis_kt<4>(s, ctas, smem, m, cols, q, k, rest...);
    case 5: return launch_basis_kt<5>(s, ctas, smem, m, cols, q, k, rest...);
    case 6: return launch_basis_kt<6>(s, ctas, smem, m, cols, q, k, rest...);
    case 7: return launch_basis_kt<7>(s, ctas, smem, m, cols, q, k, rest...);
    default: return launch_basis_kt<8>(s, ctas, smem, m, cols, q, k, rest...);
  }
}
metis_status_t launch_factors(cudaStream_t s, const FactorsArgs& f, int n_right, int n_left) {
  const dim3 grid((unsigned)(n_right + n_left));
  const size_t smem = fr_smem(f.n_in);
#define METIS_FACTORS(KT) METIS_CUDA_TRY(metis_launch_pdl((factors_kernel<KT>), grid, dim3(256), smem, s, f, n_right)); break
  switch ((f.k + 7) / 8) {
    case 1: METIS_FACTORS(1); case 2: METIS_FACTORS(2); case 3: METIS_FACTORS(3); case 4: METIS_FACTORS(4);
    case 5: METIS_FACTORS(5); case 6: METIS_FACTORS(6); case 7: METIS_FACTORS(7); default: METIS_FACTORS(8);
  }
#undef METIS_FACTORS
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// ------------------------------------------------------------------------------------------------
// Wide sketches (k + p above MAXQ or k above 64, up to 272 / 256): the same decomposition on kernels that tile over
// the rank (bigrank.cuh).  The range finder works on a contiguous matrix - the operand itself (FULL) or its sampled
// rows gathered once (SAMPLED) - so that sketch and projection both run on the tcgen05 kernel of the broadcast
// pass, in groups of sketch columns.
struct WideWs {
  size_t amax, idx, xs, omt, zp, z, gram, gram1, l, linv, evals, evecs, ycm, scale, hsp, mp, m, basis, bs, coef, part,
      a6, b6, sign, evals2, evecs2, total;
};
constexpr int WIDE_GRAM_PARTS = 32;
constexpr int WIDE_SK = 96;                              // sketch columns per launch of the tensor-core sketch
constexpr int WIDE_PJ = 80;                              // sketch columns per launch of the tensor-core projection
constexpr int WIDE_CG = 64;                              // basis vectors per launch of the broadcast pass

WideWs wide_ws_layout(int64_t rows, int64_t cols, int k, int p, int64_t n_s, bool full) {
  WideWs w{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const int q = k + p, kp = (k + 15) / 16 * 16;
  const int64_t n_r = full ? rows : n_s;
  const int nbq = (q + WIDE_SK - 1) / WIDE_SK * WIDE_SK;
  const int64_t ldh = (n_r + 63) / 64 * 64;
  w.amax = take(256);
  w.idx = take(sizeof(int) * (size_t)n_s);
  w.xs = take(full ? 0 : sizeof(__nv_bfloat16) * (size_t)n_s * cols);
  w.omt = take(sizeof(__nv_bfloat16) * (size_t)nbq * cols);
  w.zp = take(sizeof(float) * (size_t)metis_coeff_slices(n_r, cols, nullptr) * n_r * WIDE_SK);
  w.z = take(sizeof(float) * (size_t)n_r * q);
  w.gram = take(sizeof(double) * (size_t)WIDE_GRAM_PARTS * q * q);
  w.gram1 = take(sizeof(double) * (size_t)q * q);
  w.l = take(sizeof(double) * (size_t)q * q);
  w.linv = take(sizeof(double) * (size_t)q * q);                 // inverses of the factor's diagonal blocks (fewer than q * q entries)
  w.evals = take(sizeof(double) * (size_t)q);
  w.evecs = take(sizeof(double) * (size_t)q * q);
  w.ycm = take(sizeof(double) * (size_t)metis_wide::MAXQ_WIDE * q);
  w.scale = take(sizeof(double) * (size_t)q);
  w.hsp = take(sizeof(__nv_bfloat16) * 3 * (size_t)WIDE_PJ * ldh);
  w.mp = take(sizeof(float) * (size_t)8 * cols * WIDE_PJ);
  w.m = take(sizeof(float) * (size_t)q * cols);
  w.basis = take(sizeof(float) * (size_t)k * cols);
  w.bs = take(sizeof(__nv_bfloat16) * 3 * (size_t)kp * cols);
  w.coef = take(sizeof(float) * (size_t)kp * rows);
  w.part = take(sizeof(float) * (size_t)metis_coeff_slices(rows, cols, nullptr) * rows * WIDE_CG);
  w.a6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * rows);
  w.b6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * cols);
  w.sign = take(sizeof(float) * (size_t)kp);
  w.evals2 = take(sizeof(double) * (size_t)k);
  w.evecs2 = take(sizeof(double) * (size_t)k * k);
  w.total = off;
  return w;
}

bool split_is_wide(int k, int p) { return k > 64 || k + p > MAXQ; }

metis_status_t launch_gemm64(cudaStream_t s, const metis_wide::Gemm64Args& g) {
  dim3 grid((unsigned)metis_ceil_div(g.N, 64), (unsigned)metis_ceil_div(g.M, 64));
  METIS_CUDA_TRY(metis_launch_pdl(metis_wide::gemm64_kernel, grid, dim3(256), (size_t)0, s, g)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// FP64 Gram matrix of n vectors (element (r, i) at v[r * sr + i * sv]) into gram1 (n x n), by slabs of rows
metis_status_t launch_gram64(cudaStream_t s, const float* v, int64_t n_rows, int n, int64_t sr, int64_t sv, double* parts, double* gram1,
                             const int* skip = nullptr) {
  int64_t rpp = metis_ceil_div(metis_ceil_div(n_rows, WIDE_GRAM_PARTS), metis_wide::G64_R) * metis_wide::G64_R;
  if (rpp < 64) rpp = 64;
  const int n_parts = (int)metis_ceil_div(n_rows, rpp);
  const unsigned t = (unsigned)metis_ceil_div(n, metis_wide::G64_T);
  METIS_CUDA_TRY(metis_launch_pdl(metis_wide::gram64_kernel, dim3(t, t, (unsigned)n_parts), dim3(256), (size_t)0, s, v, n_rows, n, sr, sv, rpp, parts,
                                  skip)); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(metis_launch_pdl((reduce_gram_kernel), dim3((unsigned)metis_ceil_div(n * n, 32)), dim3(128), (size_t)(0), s, (const double*)parts, n_parts, n * n, gram1,
                                  skip)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// Cholesky factor of an n x n Gram matrix: in one SM's shared memory where it fits, streamed through L2 above that
metis_status_t launch_chol_wide(cudaStream_t s, const double* g, int n, double tol_rel, double* l, double* dinv, int* perm, metis_wide::EigState* st, const int* skip,
                                int* well_conditioned) {
  using namespace metis_wide;
  if (n <= CM_MAX) METIS_CUDA_TRY(metis_launch_pdl(chol_mid_kernel, dim3(1), dim3(CW_THREADS), cm_smem(n), s, g, n, tol_rel, l, dinv, perm, st, skip, well_conditioned));
  else METIS_CUDA_TRY(metis_launch_pdl(chol_wide_kernel, dim3(1), dim3(CW_THREADS), CW_SMEM, s, g, n, tol_rel, l, dinv, perm, st, skip, well_conditioned));
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// eigen-decomposition of the n x n Gram matrix gram1 (see bigrank.cuh).  scratch: the Gram partials, free by then
// (WIDE_GRAM_PARTS n x n matrices; six are used, and the state and the permutation sit in the seventh).
template <int LANES, int R>
metis_status_t launch_jacobi_fp32(cudaStream_t s, const double* l, int n, double* x) {
  cudaLaunchConfig_t cfg = {};
  const unsigned ctas = (unsigned)((n + metis_wide::JF_COLS - 1) / metis_wide::JF_COLS);
  cfg.gridDim = dim3(ctas); cfg.blockDim = dim3(LANES * metis_wide::JF_MB); cfg.dynamicSmemBytes = metis_wide::jf_smem(LANES, R); cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  METIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, (metis_wide::jacobi_fp32_kernel<LANES, R>), l, n, x)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// factor and starting vectors of a matrix of order N_FROM ... N_TO: v, zt, tri are scratch of n x n and (tri: 3 n and the panels' 8 n)
template <int N_FROM, int N_TO, int R, int C, bool TAIL>
metis_status_t launch_tridiag(cudaStream_t s, const double* gram1, int n, double* l, int* perm, metis_wide::EigState* st, double* v, double* zt, double* tri, double* x) {
  using namespace metis_wide;
  static_assert(N_TO <= WtShape<R, C, TAIL>::N_MAX && N_TO <= WT_MAX, "rows and columns of the instance");
  static_assert(N_FROM >= 32 * (TAIL ? C : C - 1), "a lane's last column is at most 32 below the first");
  double* panels = tri + 3 * n;
  const unsigned vec = (unsigned)metis_ceil_div(n, WV_WARPS), pan = (unsigned)metis_ceil_div(metis_ceil_div(n - 2, 8), WV_WARPS);
  METIS_CUDA_TRY(metis_launch_pdl((tridiag_chol_kernel<R, C, TAIL>), dim3(2), dim3(WT_THREADS), cm_smem(n), s, gram1, n, l, perm, st, v, tri)); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(metis_launch_pdl(tridiag_vectors_kernel, dim3(vec + pan), dim3(32 * WV_WARPS), (size_t)0, s, (const double*)tri, (const double*)v, n, zt, panels)); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(metis_launch_pdl(tridiag_back_kernel, dim3((unsigned)metis_ceil_div(n, 8)), dim3(WB_THREADS), wb_smem(n), s, (const double*)zt, (const double*)v,
                                  (const double*)panels, (const double*)l, (const int*)perm, n, x)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}

metis_status_t launch_eig_wide(cudaStream_t s, const double* gram1, int n, double* scratch, double* l, double* ycm, double* evals, double* evecs) {
  if (n <= MAXQ) return launch_eig(s, gram1, n, n, evals, evecs);               // a small rank with a large oversampling
  using namespace metis_wide;
  const size_t nn = (size_t)n * n;
  double *x[2] = {scratch, scratch + nn}, *w = scratch + 2 * nn, *sm = scratch + 3 * nn, *g1 = scratch + 4 * nn, *e = scratch + 5 * nn;
  EigState* st = reinterpret_cast<EigState*>(scratch + 6 * nn);
  int* failed = reinterpret_cast<int*>(st + 1);
  int* perm = failed + 1;
  if (n <= 90) METIS_TRY((launch_tridiag<MAXQ + 1, 90, 6, 3, false>(s, gram1, n, l, perm, st, w, sm, g1, x[0])));
  else if (n <= 96) METIS_TRY((launch_tridiag<91, 96, 9, 3, false>(s, gram1, n, l, perm, st, w, sm, g1, x[0])));
  else if (n <= 128) METIS_TRY((launch_tridiag<97, 128, 9, 4, false>(s, gram1, n, l, perm, st, w, sm, g1, x[0])));
  else if (n <= WT_MAX) METIS_TRY((launch_tridiag<129, WT_MAX, 10, 4, true>(s, gram1, n, l, perm, st, w, sm, g1, x[0])));
  else {
    METIS_TRY(launch_chol_wide(s, gram1, n, 1e-14, l, nullptr, perm, st, nullptr, nullptr));
    if (n <= 176) METIS_TRY((launch_jacobi_fp32<8, 22>(s, l, n, x[0])));
    else if (n <= 192) METIS_TRY((launch_jacobi_fp32<16, 12>(s, l, n, x[0])));
    else if (n <= 224) METIS_TRY((launch_jacobi_fp32<16, 14>(s, l, n, x[0])));
    else if (n <= 256) METIS_TRY((launch_jacobi_fp32<16, 16>(s, l, n, x[0])));
    else METIS_TRY((launch_jacobi_fp32<16, 18>(s, l, n, x[0])));
  }
  const unsigned t = (unsigned)((n + 31) / 32);
  for (int step = 0; step < ER_STEPS; ++step) {
    double *xc = x[step & 1], *xn = x[(step & 1) ^ 1];
    METIS_CUDA_TRY(metis_launch_pdl((refine_product_kernel<0>), dim3(t, t), dim3(128), (size_t)0, s, (const double*)l, (const double*)xc, w, (const double*)nullptr,
                                    (double*)nullptr, n, (const EigState*)st, step)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl((refine_product_kernel<1>), dim3(t, t, 2), dim3(128), (size_t)0, s, (const double*)w, (const double*)w, sm, (const double*)xc, g1, n,
                                    (const EigState*)st, step)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl(refine_correction_kernel, dim3((unsigned)((nn + 255) / 256)), dim3(256), (size_t)0, s, (const double*)sm, (const double*)g1, e, n, st,
                                    step)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl((refine_product_kernel<2>), dim3(t, t), dim3(128), (size_t)0, s, (const double*)xc, (const double*)e, xn, (const double*)nullptr,
                                    (double*)nullptr, n, (const EigState*)st, step)); METIS_COUNT_LAUNCH();
  }
  METIS_CUDA_TRY(metis_launch_pdl(eigen_finish_kernel, dim3(1), dim3(1024), (size_t)0, s, (const double*)x[0], (const double*)x[1], (const double*)sm, (const double*)g1,
                                  (const int*)perm, n, (const EigState*)st, evals, evecs, failed)); METIS_COUNT_LAUNCH();
  jacobi_cluster_kernel<<<JC_P, JC_THREADS, JC_SMEM, s>>>(l, n, 1e-12f, failed, ycm); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  jacobi_collect_kernel<<<1, 1024, 0, s>>>(ycm, n, perm, failed, evals, evecs); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  return METIS_OK;
}

metis_status_t split_wide(metis_context* ctx, const __nv_bfloat16* x, int64_t rows, int64_t cols, int k, int p, bool full, int64_t n_s,
                          uint64_t seed, int rounding, bool want_c, bool want_r, const float* src_amax, metis_operand_t* out, float* residual_dense,
                          unsigned char* wsb, const WideWs& L, cudaStream_t s) {
  using namespace metis_qt;
  using metis_wide::Gemm64Args;
  const int q = k + p, kp = (k + 15) / 16 * 16, kx6 = metis_residual_kx(kp);
  const int64_t n_r = full ? rows : n_s;
  const int64_t ldh = (n_r + 63) / 64 * 64;
  float* amax = reinterpret_cast<float*>(wsb + L.amax);
  int* idx = reinterpret_cast<int*>(wsb + L.idx);
  __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(wsb + L.xs);
  __nv_bfloat16* omt = reinterpret_cast<__nv_bfloat16*>(wsb + L.omt);
  float* zp = reinterpret_cast<float*>(wsb + L.zp);
  float* z = reinterpret_cast<float*>(wsb + L.z);
  double* gram = reinterpret_cast<double*>(wsb + L.gram);
  double* gram1 = reinterpret_cast<double*>(wsb + L.gram1);
  double* lf = reinterpret_cast<double*>(wsb + L.l);
  double* linv = reinterpret_cast<double*>(wsb + L.linv);
  double* evals = reinterpret_cast<double*>(wsb + L.evals);
  double* evecs = reinterpret_cast<double*>(wsb + L.evecs);
  double* ycm = reinterpret_cast<double*>(wsb + L.ycm);
  double* scale = reinterpret_cast<double*>(wsb + L.scale);
  __nv_bfloat16* hsp = reinterpret_cast<__nv_bfloat16*>(wsb + L.hsp);
  float* mp = reinterpret_cast<float*>(wsb + L.mp);
  float* m = reinterpret_cast<float*>(wsb + L.m);
  float* basis = reinterpret_cast<float*>(wsb + L.basis);
  __nv_bfloat16* bs = reinterpret_cast<__nv_bfloat16*>(wsb + L.bs);
  float* coef = reinterpret_cast<float*>(wsb + L.coef);
  float* part = reinterpret_cast<float*>(wsb + L.part);
  __nv_bfloat16* a6 = reinterpret_cast<__nv_bfloat16*>(wsb + L.a6);
  __nv_bfloat16* b6 = reinterpret_cast<__nv_bfloat16*>(wsb + L.b6);
  float* sign = reinterpret_cast<float*>(wsb + L.sign);
  double* evals2 = reinterpret_cast<double*>(wsb + L.evals2);
  double* evecs2 = reinterpret_cast<double*>(wsb + L.evecs2);

  METIS_CUDA_TRY(cudaMemsetAsync(amax, 0, 64, s));
  if (src_amax != nullptr) METIS_CUDA_TRY(cudaMemcpyAsync(amax, src_amax, sizeof(float), cudaMemcpyDeviceToDevice, s));
  const __nv_bfloat16* xr = x;
  if (!full) {
    METIS_CUDA_TRY(metis_launch_pdl((sample_rows_kernel), dim3((unsigned)metis_ceil_div(n_s, 256)), dim3(256), (size_t)(0), s, idx, (int)n_s, rows, seed, 0,
                                    (float*)nullptr, (unsigned long long*)nullptr)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::gather_rows_kernel, dim3((unsigned)metis_ceil_div(n_s * (cols / 8), 256)), dim3(256), (size_t)0, s, x, cols,
                                    (const int*)idx, (int)n_s, xs)); METIS_COUNT_LAUNCH();
    xr = xs;
  }
  // (2) sketch Z = xr Omega on the tensor cores, WIDE_SK sketch columns per launch
  const int nbq = (q + WIDE_SK - 1) / WIDE_SK * WIDE_SK;
  {
    const uint64_t blocks = ((uint64_t)cols * q + 7) / 8;
    METIS_CUDA_TRY(metis_launch_pdl((omega_rows_kernel), dim3((unsigned)metis_ceil_div((int64_t)blocks, 256)), dim3(256), (size_t)(0), s, cols, q, nbq, seed, ctx->quantile_lut, omt)); METIS_COUNT_LAUNCH();
    const int slices = metis_coeff_slices(n_r, cols, nullptr);
    for (int j0 = 0; j0 < q; j0 += WIDE_SK) {
      const int qg = q - j0 < WIDE_SK ? q - j0 : WIDE_SK;
      METIS_TRY(metis_launch_coeff_tc(ctx, xr, n_r, cols, omt + (int64_t)j0 * cols, WIDE_SK / 3, zp, (full && j0 == 0) ? amax : nullptr, 1, s));
      METIS_CUDA_TRY(metis_launch_pdl((reduce_sketch_kernel), dim3((unsigned)metis_ceil_div(n_r * qg, 256)), dim3(256), (size_t)(0), s, (const float*)zp, slices, n_r, WIDE_SK, qg,
                                      z + j0, q)); METIS_COUNT_LAUNCH();
    }
  }
  // (3) CholeskyQR (FP64 Gram matrix, blocked factorisation, blocked triangular solve).  The first factorisation
  // reports whether its smallest pivot is above 1e-8 of the largest diagonal entry; if so H is orthonormal to FP32
  // rounding already and the kernels of the second pass return at once.
  {
    float* src = z;
    int* cond_flag = reinterpret_cast<int*>(amax + 8);
    for (int pass = 0; pass < 2; ++pass) {
      const int* skip = pass ? cond_flag : nullptr;
      METIS_TRY(launch_gram64(s, src, n_r, q, q, 1, gram, gram1, skip));
      METIS_TRY(launch_chol_wide(s, gram1, q, 1e-13, lf, linv, nullptr, nullptr, skip, pass ? nullptr : cond_flag));
      METIS_CUDA_TRY(metis_launch_pdl(metis_wide::trsm_wide_kernel, dim3((unsigned)metis_ceil_div(n_r, metis_wide::TW_ROWS)), dim3(256), metis_wide::TW_SMEM, s, src, n_r, q,
                                      (const double*)lf, (const double*)linv, skip)); METIS_COUNT_LAUNCH();
    }
  }                                                      // H = Z L^-T, in place
  // (4) M = H^T xr on the tensor cores, WIDE_PJ sketch columns per launch; eigen-decomposition of M M^T
  {
    const int slices = metis_project_slices(n_r, cols);
    for (int j0 = 0; j0 < q; j0 += WIDE_PJ) {
      const int qg = q - j0 < WIDE_PJ ? q - j0 : WIDE_PJ;
      const int jp = (qg + 15) / 16 * 16;
      METIS_CUDA_TRY(metis_launch_pdl(h_splits_kernel, dim3((unsigned)metis_ceil_div(ldh, 256), (unsigned)jp), dim3(256), (size_t)0, s, (const float*)(z + j0), (int)n_r, qg, jp,
                                      (int)ldh, hsp, q)); METIS_COUNT_LAUNCH();
      METIS_TRY(metis_launch_project_tc(ctx, xr, n_r, cols, hsp, jp, ldh, mp, s));
      dim3 rgrid((unsigned)metis_ceil_div(cols, 32), (unsigned)metis_ceil_div(qg, 32));
      METIS_CUDA_TRY(metis_launch_pdl((reduce_proj_kernel), rgrid, dim3(256), (size_t)(0), s, (const float*)mp, slices, cols, jp, qg, m + (int64_t)j0 * cols)); METIS_COUNT_LAUNCH();
    }
    METIS_TRY(launch_gram64(s, m, cols, q, 1, cols, gram, gram1));
    METIS_TRY(launch_eig_wide(s, gram1, q, gram, lf, ycm, evals, evecs));
  }
  // right basis: basis[j][col] = sum_i evecs[i][j] M[i][col] / sqrt(eval_j),  j < k
  float* rb = full ? out->right : basis;
  {
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::rot_scales_kernel, dim3((unsigned)metis_ceil_div(k, 128)), dim3(128), (size_t)0, s, (const double*)evals, (const float*)nullptr, k, 0,
                                    scale, full ? out->sigma : (float*)nullptr)); METIS_COUNT_LAUNCH();
    Gemm64Args g{};
    g.a = m; g.a_m = 1; g.a_k = cols; g.b = evecs; g.b_k = q; g.b_n = 1; g.scale = scale; g.c = rb; g.c_m = 1; g.c_n = cols; g.M = cols; g.N = k; g.K = q;
    METIS_TRY(launch_gemm64(s, g));
  }
  QuantParams qp{};
  metis_nvfp4_t rc = out->res_by_cols, rr = out->res_by_rows;
  rc.rows = rows; rc.k_len = cols; rr.rows = cols; rr.k_len = rows;
  qp.rows = rows; qp.cols = cols; qp.rounding = rounding; qp.seed = seed; qp.stream_id = METIS_STREAM_RESIDUAL;
  qp.e_stride_r = cols; qp.e_stride_c = 1;
  if (want_c) { qp.c_codes = rc.codes; qp.c_scales = rc.scales; qp.c_layout = rc.sf_layout; }
  if (want_r) { qp.r_codes = rr.codes; qp.r_scales = rr.scales; qp.r_layout = rr.sf_layout; }
  float* t0 = want_c ? rc.tensor_scale : nullptr; float* t1 = want_r ? rr.tensor_scale : nullptr;
  const dim3 bs_grid((unsigned)metis_ceil_div(cols, 128), (unsigned)(kp / 8));
  cudaStream_t sf = ctx->side[0];
  if (full) {
    // right = basis with the sign convention, left = H U~_k (same flips), coefficients = left * sigma
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::sign_rows_kernel, dim3((unsigned)k), dim3(256), (size_t)0, s, out->right, cols, sign, amax + 2)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl((basis_splits_kernel), bs_grid, dim3(128), (size_t)(0), s, (const float*)out->right, cols, k, kp, bs, b6, kx6)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::rot_scales_kernel, dim3((unsigned)metis_ceil_div(k, 128)), dim3(128), (size_t)0, s, (const double*)evals, (const float*)sign, k, 2,
                                    scale, (float*)nullptr)); METIS_COUNT_LAUNCH();
    if (kp > k) METIS_CUDA_TRY(cudaMemsetAsync(coef, 0, sizeof(float) * (size_t)kp * rows, s));
    Gemm64Args g{};
    g.a = z; g.a_m = q; g.a_k = 1; g.b = evecs; g.b_k = q; g.b_n = 1; g.scale = scale; g.c = out->left; g.c_m = 1; g.c_n = rows;
    g.c2 = coef; g.c2_m = kp; g.c2_n = 1; g.scale2 = out->sigma; g.amax = amax + 1; g.M = rows; g.N = k; g.K = q;
    METIS_TRY(launch_gemm64(s, g));
    METIS_TRY(metis_fork(ctx, s, 1));
    METIS_TRY(metis_launch_residual_tc(ctx, x, coef, k, kp, qp, amax, t0, t1, residual_dense, a6, b6, s));
  } else {
    METIS_CUDA_TRY(metis_launch_pdl((basis_splits_kernel), bs_grid, dim3(128), (size_t)(0), s, (const float*)basis, cols, k, kp, bs, b6, kx6)); METIS_COUNT_LAUNCH();
    // (5) broadcast C = x B, WIDE_CG basis vectors per pass over x
    const int slices = metis_coeff_slices(rows, cols, nullptr);
    for (int j0 = 0; j0 < kp; j0 += WIDE_CG) {
      const int gw = kp - j0 < WIDE_CG ? kp - j0 : WIDE_CG;
      METIS_TRY(metis_launch_coeff_tc(ctx, x, rows, cols, bs + (int64_t)3 * j0 * cols, gw, part, j0 == 0 ? amax : nullptr, 0, s));
      METIS_CUDA_TRY(metis_launch_pdl(metis_wide::coef_sum_kernel, dim3((unsigned)metis_ceil_div(rows * (gw / 8), 256)), dim3(256), (size_t)0, s, (const float*)part, slices, rows, gw, j0,
                                      kp, coef, a6, kx6)); METIS_COUNT_LAUNCH();
    }
    METIS_TRY(metis_fork(ctx, s, 1));
    METIS_TRY(metis_launch_residual_tc(ctx, x, nullptr, k, kp, qp, amax, t0, t1, residual_dense, a6, b6, s));
    // (7) Rayleigh-Ritz on C^T C, rotate both factors (side stream, beside the residual pass)
    METIS_TRY(launch_gram64(sf, coef, rows, k, kp, 1, gram, gram1));
    METIS_TRY(launch_eig_wide(sf, gram1, k, gram, lf, ycm, evals2, evecs2));
    {
      Gemm64Args g{};
      g.a = basis; g.a_m = 1; g.a_k = cols; g.b = evecs2; g.b_k = k; g.b_n = 1; g.c = out->right; g.c_m = 1; g.c_n = cols; g.M = cols; g.N = k; g.K = k;
      METIS_TRY(launch_gemm64(sf, g));
    }
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::sign_rows_kernel, dim3((unsigned)k), dim3(256), (size_t)0, sf, out->right, cols, sign, amax + 2)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::rot_scales_kernel, dim3((unsigned)metis_ceil_div(k, 128)), dim3(128), (size_t)0, sf, (const double*)evals2, (const float*)sign, k, 1,
                                    scale, out->sigma)); METIS_COUNT_LAUNCH();
    {
      Gemm64Args g{};
      g.a = coef; g.a_m = kp; g.a_k = 1; g.b = evecs2; g.b_k = k; g.b_n = 1; g.scale = scale; g.c = out->left; g.c_m = 1; g.c_n = rows; g.amax = amax + 1;
      g.M = rows; g.N = k; g.K = k;
      METIS_TRY(launch_gemm64(sf, g));
    }
  }
  METIS_CUDA_TRY(metis_launch_pdl((split_status_kernel), dim3(1), dim3(32), (size_t)(0), s, (const float*)amax, (const double*)evals, k, ctx->dev_status)); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  metis_nvfp4_t lq = out->left_q, rq = out->right_q;
  lq.rows = k; lq.k_len = rows; rq.rows = k; rq.k_len = cols;
  METIS_TRY(metis_launch_quantize_factors(out->left, rows, out->right, cols, k, rounding, seed, amax + 1, amax + 2, &lq, &rq, sf));
  return metis_join(ctx, s, 0);
}

}  // namespace

metis_status_t metis_debug_eigen(metis_handle_t h, const double* gram, int32_t n, double* evals, double* evecs, void* ws, size_t ws_bytes, metis_stream_t stream) {
  if (!h || !gram || !evals || !evecs) return METIS_ERR_INVALID_ARG;
  if (n < 1 || n > metis_wide::MAXQ_WIDE) return METIS_ERR_SHAPE;
  const size_t nn = (size_t)n * n;
  if (n > MAXQ && (!ws || !metis_aligned16(ws) || ws_bytes < sizeof(double) * (8 * nn + (size_t)metis_wide::MAXQ_WIDE * n))) return METIS_ERR_WORKSPACE;
  double* scratch = reinterpret_cast<double*>(ws);        // seven matrices, then the factor and the columns of the FP64 sweeps
  return launch_eig_wide(reinterpret_cast<cudaStream_t>(stream), gram, n, scratch, scratch + 7 * nn, scratch + 8 * nn, evals, evecs);
}

int64_t metis_default_sample_count(int64_t rows, int32_t q) {
  int64_t want = 4 * (int64_t)q;
  const int64_t pct = (rows + 99) / 100;
  if (pct > want) want = pct;
  want = (want + 15) / 16 * 16;
  return want < rows ? want : rows;
}

metis_status_t metis_split_set_attrs() {
#define METIS_OA_ATTR(KT) METIS_CUDA_TRY(cudaFuncSetAttribute(orth_apply_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)oa_smem(KT)))
  METIS_OA_ATTR(1); METIS_OA_ATTR(2); METIS_OA_ATTR(3); METIS_OA_ATTR(4); METIS_OA_ATTR(5); METIS_OA_ATTR(6); METIS_OA_ATTR(7); METIS_OA_ATTR(8); METIS_OA_ATTR(9);
#undef METIS_OA_ATTR
  METIS_CUDA_TRY(cudaFuncSetAttribute(chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CHOL_SMEM));
#define METIS_FR_ATTR(KT) METIS_CUDA_TRY(cudaFuncSetAttribute(basis_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fr_smem(MAXQ))); \
  METIS_CUDA_TRY(cudaFuncSetAttribute(factors_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fr_smem(MAXQ)))
  METIS_FR_ATTR(1); METIS_FR_ATTR(2); METIS_FR_ATTR(3); METIS_FR_ATTR(4); METIS_FR_ATTR(5); METIS_FR_ATTR(6); METIS_FR_ATTR(7); METIS_FR_ATTR(8);
#undef METIS_FR_ATTR
#define METIS_EIG_ATTR(NT8) METIS_CUDA_TRY(cudaFuncSetAttribute(metis_small::eig_kernel<NT8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_small::eig_smem(8 * NT8)))
  METIS_EIG_ATTR(1); METIS_EIG_ATTR(2); METIS_EIG_ATTR(3); METIS_EIG_ATTR(4); METIS_EIG_ATTR(5); METIS_EIG_ATTR(6); METIS_EIG_ATTR(7); METIS_EIG_ATTR(8); METIS_EIG_ATTR(9);
#undef METIS_EIG_ATTR
  METIS_CUDA_TRY(cudaFuncSetAttribute(gram_chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)GC_MAX_SMEM));
  METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::jacobi_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::JC_SMEM));
#define METIS_WT_ATTR(R, C, T) METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::tridiag_chol_kernel<R, C, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::cm_smem(metis_wide::WT_MAX)))
  METIS_WT_ATTR(6, 3, false); METIS_WT_ATTR(9, 3, false); METIS_WT_ATTR(9, 4, false); METIS_WT_ATTR(10, 4, true);
#undef METIS_WT_ATTR
  METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::tridiag_back_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::wb_smem(metis_wide::WT_MAX)));
#define METIS_JF_ATTR(LN, R) METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::jacobi_fp32_kernel<LN, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::jf_smem(LN, R)))
  METIS_JF_ATTR(8, 22);
  METIS_JF_ATTR(16, 12); METIS_JF_ATTR(16, 14); METIS_JF_ATTR(16, 16); METIS_JF_ATTR(16, 18);
#undef METIS_JF_ATTR
  METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::chol_mid_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::cm_smem(metis_wide::CM_MAX)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::chol_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::CW_SMEM));
  METIS_CUDA_TRY(cudaFuncSetAttribute(metis_wide::trsm_wide_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_wide::TW_SMEM));
#define METIS_PP_ATTR(MTV) METIS_CUDA_TRY(cudaFuncSetAttribute(project_pipe_kernel<MTV>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
      (int)((size_t)PP_STAGES * (PP_K * PP_XP * 2 + 3 * (MTV) * 16 * PP_HP * 2))))
  METIS_PP_ATTR(1); METIS_PP_ATTR(2); METIS_PP_ATTR(3); METIS_PP_ATTR(4); METIS_PP_ATTR(5);
#undef METIS_PP_ATTR
  return METIS_OK;
}

// flags METIS_DEV_NONFINITE when *amax (the amax of a tensor about to be quantized) is not a finite number
metis_status_t metis_launch_amax_check(metis_context* ctx, const float* amax, cudaStream_t s) {
  METIS_CUDA_TRY(metis_launch_pdl((split_status_kernel), dim3(1), dim3(32), (size_t)(0), s, amax, (const double*)nullptr, 0, ctx->dev_status));
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

namespace {
// contiguous BF16 copy of a strided BF16 or FP32 operand (FP32 rounded to nearest even), eight elements per thread
__global__ void __launch_bounds__(256)
pack_bf16_kernel(const void* __restrict__ x, int dtype, int64_t rows, int64_t cols, int64_t ld, __nv_bfloat16* __restrict__ out) {
  metis_pdl_wait_trigger();
  const int64_t g = (int64_t)blockIdx.x * 256 + threadIdx.x, per_row = cols / 8;
  if (g >= rows * per_row) return;
  const int64_t r = g / per_row, c = (g - r * per_row) * 8;
  uint4 o;
  if (dtype == METIS_BF16) {
    o = *reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(x) + r * ld + c);
  } else {
    const float4* src = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(x) + r * ld + c);
    const float4 a = src[0], b = src[1];
    __nv_bfloat162 h0 = __floats2bfloat162_rn(a.x, a.y), h1 = __floats2bfloat162_rn(a.z, a.w);
    __nv_bfloat162 h2 = __floats2bfloat162_rn(b.x, b.y), h3 = __floats2bfloat162_rn(b.z, b.w);
    o.x = *reinterpret_cast<uint32_t*>(&h0); o.y = *reinterpret_cast<uint32_t*>(&h1);
    o.z = *reinterpret_cast<uint32_t*>(&h2); o.w = *reinterpret_cast<uint32_t*>(&h3);
  }
  *reinterpret_cast<uint4*>(out + r * cols + c) = o;
}
metis_status_t launch_pack_bf16(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, __nv_bfloat16* out, cudaStream_t s) {
  METIS_CUDA_TRY(metis_launch_pdl(pack_bf16_kernel, dim3((unsigned)metis_ceil_div(rows * (cols / 8), 256)), dim3(256), (size_t)0, s, x, dtype, rows, cols, ld, out));
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}
}  // namespace

size_t metis_split_ws_bytes(int64_t rows, int64_t cols, int k, int p) {
  if (k > 0 && split_is_wide(k, p)) {
    // the larger of the FULL layout and the SAMPLED layout with the default sample count
    const size_t a = wide_ws_layout(rows, cols, k, p, rows, true).total;
    const size_t b = wide_ws_layout(rows, cols, k, p, metis_default_sample_count(rows, k + p), false).total;
    return a > b ? a : b;
  }
  // Every buffer grows with the sample count except the sketch partials, whose chunk width steps from 64 to 256
  // columns above 512 sampled rows: the FULL sketch (n_s = rows) and a 512-row sample bound every other case.
  const size_t full = split_ws_layout(rows, cols, k, p, rows).total;
  const size_t narrow = split_ws_layout(rows, cols, k, p, rows < 512 ? rows : 512).total;
  return full > narrow ? full : narrow;
}

metis_status_t metis_split(metis_handle_t h, const void* xv, int32_t dtype, int64_t rows, int64_t cols, int64_t ld, int32_t k, int32_t p,
                           int32_t sketch, int64_t n_sample, uint64_t seed, int32_t rounding, int32_t residual_axes,
                           const float* src_amax, metis_operand_t* out, float* residual_dense, void* ws, size_t ws_bytes,
                           metis_stream_t stream) {
  METIS_NVTX("metis_split");
  using namespace metis_qt;
  if (!h || !xv || !out || !ws) return METIS_ERR_INVALID_ARG;
  if (dtype != METIS_BF16 && dtype != METIS_FP32) return METIS_ERR_INVALID_ARG;
  if (rows <= 0 || cols <= 0 || rows % 16 || cols % 16 || k < 0 || p < 0 || ld < cols) return METIS_ERR_SHAPE;
  if (ld % (dtype == METIS_BF16 ? 8 : 4)) return METIS_ERR_ALIGNMENT;          // every row starts on a 16-byte boundary
  // anything but a contiguous BF16 operand is packed (and rounded) into the tail of the workspace first
  const bool packed = k > 0 && (dtype != METIS_BF16 || ld != cols);
  const size_t pack_bytes = packed ? (((size_t)rows * (size_t)cols * sizeof(__nv_bfloat16) + 255) & ~(size_t)255) : 0;
  if (k > 0 && (k > metis_wide::MAXK_WIDE || k + p > metis_wide::MAXQ_WIDE || k % 4)) return METIS_ERR_SHAPE;
  const bool wide = k > 0 && split_is_wide(k, p);
  if (out->k != k || out->rows != rows || out->cols != cols) return METIS_ERR_INVALID_ARG;
  if (!metis_aligned16(xv) || !metis_aligned16(ws)) return METIS_ERR_ALIGNMENT;
  if (rounding != METIS_ROUND_RNE && rounding != METIS_ROUND_SR) return METIS_ERR_INVALID_ARG;
  if (sketch != METIS_SKETCH_FULL && sketch != METIS_SKETCH_SAMPLED) return METIS_ERR_INVALID_ARG;
  const bool want_c = (residual_axes & METIS_BLOCKS_ALONG_COLS) != 0, want_r = (residual_axes & METIS_BLOCKS_ALONG_ROWS) != 0;
  if (want_c && (!out->res_by_cols.codes || !out->res_by_cols.scales || !out->res_by_cols.tensor_scale)) return METIS_ERR_INVALID_ARG;
  if (want_r && (!out->res_by_rows.codes || !out->res_by_rows.scales || !out->res_by_rows.tensor_scale)) return METIS_ERR_INVALID_ARG;
  if (want_c && out->res_by_cols.sf_layout == METIS_SF_TILED && cols % 64) return METIS_ERR_SHAPE;
  if (want_r && out->res_by_rows.sf_layout == METIS_SF_TILED && rows % 64) return METIS_ERR_SHAPE;
  const int q = k + p;
  const bool full = sketch == METIS_SKETCH_FULL;
  int64_t n_s = full ? rows : (n_sample > 0 ? n_sample : metis_default_sample_count(rows, q));
  if (k > 0 && (n_s > rows || n_s % 16 || q > n_s || q > cols)) return METIS_ERR_SHAPE;
  if (k == 0) n_s = 16;
  if (wide) {
    // the tensor-core passes carry the wide path: 16-byte aligned rows of x, whole 64-column chunks
    if (cols % 64 || rows % 64) return METIS_ERR_SHAPE;
    const WideWs W = wide_ws_layout(rows, cols, k, p, n_s, full);
    if (ws_bytes < W.total + pack_bytes) return METIS_ERR_WORKSPACE;
    if (!out->left || !out->sigma || !out->right || !out->left_q.codes || !out->right_q.codes || !out->left_q.scales ||
        !out->right_q.scales || !out->left_q.tensor_scale || !out->right_q.tensor_scale)
      return METIS_ERR_INVALID_ARG;
    const __nv_bfloat16* xw = reinterpret_cast<const __nv_bfloat16*>(xv);
    if (packed) {
      __nv_bfloat16* xp = reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<unsigned char*>(ws) + ((W.total + 255) & ~(size_t)255));
      METIS_TRY(launch_pack_bf16(xv, dtype, rows, cols, ld, xp, reinterpret_cast<cudaStream_t>(stream)));
      xw = xp;
    }
    return split_wide(h, xw, rows, cols, k, p, full, n_s, seed, rounding, want_c, want_r, src_amax, out,
                      residual_dense, reinterpret_cast<unsigned char*>(ws), W, reinterpret_cast<cudaStream_t>(stream));
  }
  const SplitWs L = split_ws_layout(rows, cols, k, p, n_s);
  if (ws_bytes < L.total + pack_bytes) return METIS_ERR_WORKSPACE;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  unsigned char* wsb = reinterpret_cast<unsigned char*>(ws);
  const __nv_bfloat16* x = reinterpret_cast<const __nv_bfloat16*>(xv);
  if (packed) {
    __nv_bfloat16* xp = reinterpret_cast<__nv_bfloat16*>(wsb + ((L.total + 255) & ~(size_t)255));
    METIS_TRY(launch_pack_bf16(xv, dtype, rows, cols, ld, xp, s));
    x = xp;
  }
  float* amax = reinterpret_cast<float*>(wsb + L.amax);

  metis_nvfp4_t rc = out->res_by_cols, rr = out->res_by_rows;
  rc.rows = rows; rc.k_len = cols; rr.rows = cols; rr.k_len = rows;
  if (k == 0) {
    if (src_amax != nullptr) METIS_CUDA_TRY(cudaMemcpyAsync(amax, src_amax, sizeof(float), cudaMemcpyDeviceToDevice, s));
    else METIS_TRY(metis_launch_amax(xv, dtype, rows, cols, ld, amax, s));
    METIS_TRY(metis_launch_quantize(xv, dtype, rows, cols, ld, rounding, seed, METIS_STREAM_RESIDUAL, cols, 1, amax,
                                    1, want_c ? &rc : nullptr, want_r ? &rr : nullptr, s, h->dev_status));
    return METIS_OK;
  }
  if (!out->left || !out->sigma || !out->right || !out->left_q.codes || !out->right_q.codes || !out->left_q.scales ||
      !out->right_q.scales || !out->left_q.tensor_scale || !out->right_q.tensor_scale)
    return METIS_ERR_INVALID_ARG;
  if (out->left_q.sf_layout == METIS_SF_TILED && rows % 64) return METIS_ERR_SHAPE;
  if (out->right_q.sf_layout == METIS_SF_TILED && cols % 64) return METIS_ERR_SHAPE;

  int* idx = reinterpret_cast<int*>(wsb + L.idx);
  float* zp = reinterpret_cast<float*>(wsb + L.zp);
  float* z = reinterpret_cast<float*>(wsb + L.z);
  double* gram = reinterpret_cast<double*>(wsb + L.gram);
  double* linvt = reinterpret_cast<double*>(wsb + L.linv);
  int* cond_flag = reinterpret_cast<int*>(amax + 8);
  double* gram1 = reinterpret_cast<double*>(wsb + L.gram1);
  double* evals = reinterpret_cast<double*>(wsb + L.evals);
  double* evecs = reinterpret_cast<double*>(wsb + L.evecs);
  float* mp = reinterpret_cast<float*>(wsb + L.mp);
  float* m = reinterpret_cast<float*>(wsb + L.m);
  float* basis = reinterpret_cast<float*>(wsb + L.basis);
  float* coef = reinterpret_cast<float*>(wsb + L.coef);
  unsigned long long* keys = reinterpret_cast<unsigned long long*>(wsb + L.keys);          // sign contest, one per vector
  double* evals2 = reinterpret_cast<double*>(wsb + L.evals2);
  double* evecs2 = reinterpret_cast<double*>(wsb + L.evecs2);
  __nv_bfloat16* bs = reinterpret_cast<__nv_bfloat16*>(wsb + L.bs);
  double* gram_c = reinterpret_cast<double*>(wsb + L.gram_c);
  float* part = reinterpret_cast<float*>(wsb + L.part);
  __nv_bfloat16* hsp = reinterpret_cast<__nv_bfloat16*>(wsb + L.hsp);
  __nv_bfloat16* a6 = reinterpret_cast<__nv_bfloat16*>(wsb + L.a6);
  __nv_bfloat16* b6 = reinterpret_cast<__nv_bfloat16*>(wsb + L.b6);
  // the residual kernel's K-concatenated BF16 operands are written by the kernels that produce coefficients and basis
  const int kx6 = metis_residual_kx((k + 15) / 16 * 16);
  metis_context* ctx = h;
  const int kp = (k + 15) / 16 * 16;
  // (1) row sample (clears the amax slots of x, left and right, the condition flag and the sign keys), (2) sketch (tensor cores; Omega
  // generated per CTA into shared memory).  amax|x| for the residual's tensor scale: fused into the sketch pass (FULL) or
  // the broadcast pass (SAMPLED).
  METIS_CUDA_TRY(metis_launch_pdl((sample_rows_kernel), dim3((unsigned)metis_ceil_div(n_s, 256)), dim3(256), (size_t)(0), s, idx, (int)n_s, rows, seed, full ? 1 : 0, amax, keys)); METIS_COUNT_LAUNCH();
  if (src_amax != nullptr) METIS_CUDA_TRY(cudaMemcpyAsync(amax, src_amax, sizeof(float), cudaMemcpyDeviceToDevice, s));
  const int ccols = sketch_chunk_cols(n_s);
  const int chunks = (int)metis_ceil_div(cols, ccols);
  __nv_bfloat16* omt = reinterpret_cast<__nv_bfloat16*>(wsb + L.omt);
  const int nb_sk = sketch_tc_cols(q);
  const bool sketch_tc = full && q <= 96 && metis_coeff_tc_usable(x, omt, cols, nb_sk / 3);
  if (sketch_tc) {
    const uint64_t blocks = ((uint64_t)cols * q + 7) / 8;
    METIS_CUDA_TRY(metis_launch_pdl((omega_rows_kernel), dim3((unsigned)metis_ceil_div((int64_t)blocks, 256)), dim3(256), (size_t)(0), s, cols, q, nb_sk, seed, ctx->quantile_lut, omt)); METIS_COUNT_LAUNCH();
    METIS_TRY(metis_launch_coeff_tc(ctx, x, rows, cols, omt, nb_sk / 3, zp, amax, 1, s));
    const int slices = metis_coeff_slices(rows, cols, nullptr);
    METIS_CUDA_TRY(metis_launch_pdl((reduce_sketch_kernel), dim3((unsigned)metis_ceil_div(rows * q, 256)), dim3(256), (size_t)(0), s, zp, slices, rows, nb_sk, q, z, q)); METIS_COUNT_LAUNCH();
  } else {
    const int nt = (q + 7) / 8;
    const size_t smem = sizeof(__nv_bfloat16) * nt * 8 * SKM_PITCH;
    dim3 grid((unsigned)metis_ceil_div(n_s, SKM_ROWS), (unsigned)chunks);
    float* am = full ? amax : nullptr;                  // FULL mode: amax|x| comes out of this pass
    switch (nt) {
      case 1: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<1>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 2: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<2>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 3: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<3>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 4: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<4>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 5: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<5>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 6: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<6>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 7: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<7>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      case 8: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<8>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
      default: METIS_CUDA_TRY(metis_launch_pdl((sketch_mma_kernel<9>), dim3(grid), dim3(256), (size_t)(smem), s, x, cols, idx, (int)n_s, q, seed, ctx->quantile_lut, zp, am, ccols)); break;
    }
    METIS_COUNT_LAUNCH();
  }
  if (!sketch_tc) {
    METIS_CUDA_TRY(metis_launch_pdl((reduce_partials_kernel), dim3((unsigned)metis_ceil_div(n_s * q, 256)), dim3(256), (size_t)(0), s, zp, chunks, n_s * q, z)); METIS_COUNT_LAUNCH();
  }
  // (3) CholeskyQR2: orthonormal basis H of range(Z), in place
  // the projection on tensor cores wants the BF16 splits of H as well (n_s >= 1024)
  const bool split_h = n_s >= 1024 && cols % 8 == 0, one_cta = gram_chol_smem(n_s, q) <= GC_MAX_SMEM;
  const int jp = (q + 15) / 16 * 16, ldh = (int)((n_s + 63) / 64 * 64);
  if (one_cta) {
    // a short sketch: Gram matrix and factorisation in one CTA; the product with L^-T on many CTAs unless the sketch
    // was ill-conditioned, in which case the first kernel has done both passes itself and the second returns at once
    METIS_CUDA_TRY(metis_launch_pdl((gram_chol_kernel), dim3(1), dim3(GC_THREADS), gram_chol_smem(n_s, q), s, z, (int)n_s, q, linvt, cond_flag)); METIS_COUNT_LAUNCH();
    METIS_TRY(launch_orth_apply(s, z, n_s, q, linvt, cond_flag, nullptr, jp, ldh));
  } else {
    for (int pass = 0; pass < 2; ++pass) {
      int64_t rpp; const int parts = gram_parts(n_s, &rpp);
      const int* skip = pass == 0 ? nullptr : cond_flag;
      METIS_CUDA_TRY(metis_launch_pdl((gram_kernel), dim3(parts), dim3(256), (size_t)(0), s, z, n_s, q, q, 1, rpp, gram, skip)); METIS_COUNT_LAUNCH();
      METIS_CUDA_TRY(metis_launch_pdl((reduce_gram_kernel), dim3((unsigned)metis_ceil_div(q * q, 32)), dim3(128), (size_t)(0), s, gram, parts, q * q, gram1, skip)); METIS_COUNT_LAUNCH();
      METIS_CUDA_TRY(metis_launch_pdl((chol_kernel), dim3(1), dim3(512), CHOL_SMEM, s, gram1, q, linvt, skip, pass == 0 ? cond_flag : nullptr)); METIS_COUNT_LAUNCH();
      METIS_TRY(launch_orth_apply(s, z, n_s, q, linvt, skip, split_h ? hsp : nullptr, jp, ldh));
    }
  }
  // (4) M = H^T x[S,:], eigen-decomposition of M M^T, right basis
  {
    int rpp; int parts;
    bool project_tc = false;
    if (split_h) {
      if (one_cta) {                                    // that factorisation leaves the splits to a kernel of their own
        METIS_CUDA_TRY(metis_launch_pdl(h_splits_kernel, dim3((unsigned)metis_ceil_div(ldh, 256), (unsigned)jp), dim3(256), (size_t)0, s, z, (int)n_s, q, jp, ldh, hsp, q)); METIS_COUNT_LAUNCH();
      }
      parts = (int)metis_ceil_div(n_s, 512);
      if (parts > PJ_MAX_PARTS) parts = PJ_MAX_PARTS;
      rpp = (int)(metis_ceil_div(metis_ceil_div(n_s, parts), PP_K) * PP_K);
      parts = (int)metis_ceil_div(n_s, rpp);
      const int mt = jp / 16;
      project_tc = full && metis_project_tc_usable(x, hsp, cols, jp);
      if (project_tc) {
        // every row, in order: M^T = x^T H on the tcgen05 kernel of the broadcast pass (x as an MN-major operand)
        METIS_TRY(metis_launch_project_tc(ctx, x, rows, cols, hsp, jp, ldh, mp, s));
        dim3 rgrid((unsigned)metis_ceil_div(cols, 32), (unsigned)metis_ceil_div(q, 32));
        METIS_CUDA_TRY(metis_launch_pdl((reduce_proj_kernel), rgrid, dim3(256), (size_t)(0), s, mp, metis_project_slices(rows, cols), cols, jp, q, m)); METIS_COUNT_LAUNCH();
      } else {
      dim3 grid((unsigned)metis_ceil_div(cols, PP_COLS), (unsigned)parts);
      const size_t psmem = (size_t)PP_STAGES * (PP_K * PP_XP * 2 + 3 * jp * PP_HP * 2);
#define METIS_PP(MTV) { \
        METIS_CUDA_TRY(metis_launch_pdl((project_pipe_kernel<MTV>), grid, dim3(256), psmem, s, x, cols, idx, (int)n_s, q, hsp, ldh, rpp, mp)); }
      switch (mt) {
        case 1: METIS_PP(1); break;
        case 2: METIS_PP(2); break;
        case 3: METIS_PP(3); break;
        case 4: METIS_PP(4); break;
        default: METIS_PP(5); break;
      }
#undef METIS_PP
      METIS_COUNT_LAUNCH();
      }
    } else {
    parts = project_parts(n_s, cols, &rpp);
    dim3 grid((unsigned)metis_ceil_div(cols, PJ_COLS), (unsigned)parts);
    const int nj4 = (q + 7) / 8;
    switch (nj4) {
      case 1: launch_project<1>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 2: launch_project<2>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 3: launch_project<3>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 4: launch_project<4>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 5: launch_project<5>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 6: launch_project<6>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 7: launch_project<7>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      case 8: launch_project<8>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
      default: launch_project<9>(grid, s, x, cols, idx, (int)n_s, q, z, rpp, mp); break;
    }
    }
    if (!project_tc) {
      METIS_CUDA_TRY(metis_launch_pdl((reduce_partials_kernel), dim3((unsigned)metis_ceil_div((int64_t)q * cols, 256)), dim3(256), (size_t)(0), s, mp, parts, (int64_t)q * cols, m)); METIS_COUNT_LAUNCH();
    }
  }
  {
    int64_t rpp; const int parts = gram_parts(cols, &rpp);
    METIS_CUDA_TRY(metis_launch_pdl((gram_kernel), dim3(parts), dim3(256), (size_t)(0), s, m, cols, q, 1, cols, rpp, gram, nullptr)); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl((reduce_gram_kernel), dim3((unsigned)metis_ceil_div(q * q, 32)), dim3(128), (size_t)(0), s, gram, parts, q * q, gram1, nullptr)); METIS_COUNT_LAUNCH();
    METIS_TRY(launch_eig(s, gram1, q, q, evals, evecs));
  }
  // (5) right basis and its splits; coefficients of every row in the basis, (6) fused residual + quantizer
  const int n_cta_c = (int)metis_ceil_div(rows, 32);
  const int n_cta_cols = (int)metis_ceil_div(cols, FR_POS), n_cta_rows = (int)metis_ceil_div(rows, FR_POS);
  float* rb = full ? out->right : basis;
  METIS_TRY(launch_basis(s, n_cta_cols, fr_smem(q), m, cols, q, k, kp, evals, evecs, rb, full ? (__nv_bfloat16*)nullptr : bs, b6, kx6, full ? out->sigma : nullptr, full ? keys : nullptr, amax + 2));
  if (full) {
    // left = H U~_k; coefficients = left * sigma, as the residual product's operand
    FactorsArgs f{};
    f.w = evecs; f.ldw = q; f.n_in = q; f.k = k; f.kp = kp;
    f.src = z; f.ld = q; f.rows = rows; f.left = out->left; f.amax_left = amax + 1;
    f.sigma_for_coef = out->sigma; f.a6 = a6; f.kx = kx6;
    METIS_TRY(launch_factors(s, f, 0, n_cta_rows));
  } else {
    // tensor-core pass over x (column slices), then the slices are summed and the Gram partials formed
    METIS_TRY(metis_launch_coeff_tc(ctx, x, rows, cols, bs, kp, part, amax, 0, s));
    const int slices = metis_coeff_slices(rows, cols, nullptr);
    switch (kp) {
      case 16: METIS_CUDA_TRY(metis_launch_pdl((coef_finish_kernel<16>), dim3(n_cta_c), dim3(256), (size_t)(0), s, part, slices, rows, coef, gram_c, a6, kx6)); break;
      case 32: METIS_CUDA_TRY(metis_launch_pdl((coef_finish_kernel<32>), dim3(n_cta_c), dim3(256), (size_t)(0), s, part, slices, rows, coef, gram_c, a6, kx6)); break;
      case 48: METIS_CUDA_TRY(metis_launch_pdl((coef_finish_kernel<48>), dim3(n_cta_c), dim3(256), (size_t)(0), s, part, slices, rows, coef, gram_c, a6, kx6)); break;
      default: METIS_CUDA_TRY(metis_launch_pdl((coef_finish_kernel<64>), dim3(n_cta_c), dim3(256), (size_t)(0), s, part, slices, rows, coef, gram_c, a6, kx6)); break;
    }
    METIS_COUNT_LAUNCH();
  }
  {
    QuantParams qp{};
    qp.rows = rows; qp.cols = cols; qp.rounding = rounding; qp.seed = seed; qp.stream_id = METIS_STREAM_RESIDUAL;
    qp.e_stride_r = cols; qp.e_stride_c = 1;
    if (want_c) { qp.c_codes = rc.codes; qp.c_scales = rc.scales; qp.c_layout = rc.sf_layout; }
    if (want_r) { qp.r_codes = rr.codes; qp.r_scales = rr.scales; qp.r_layout = rr.sf_layout; }
    float* t0 = want_c ? rc.tensor_scale : nullptr; float* t1 = want_r ? rr.tensor_scale : nullptr;
    // the big residual pass and the small factor chain below are independent from here on: the factor chain
    // goes to a (high-priority) side stream and is joined back at the end of the call
    METIS_TRY(metis_fork(ctx, s, 1));
    METIS_TRY(metis_launch_residual_tc(ctx, x, nullptr, k, kp, qp, amax, t0, t1, residual_dense, a6, b6, s));
    METIS_CUDA_TRY(metis_launch_pdl((split_status_kernel), dim3(1), dim3(32), (size_t)(0), s, amax, evals, k, ctx->dev_status)); METIS_COUNT_LAUNCH();
  }
  cudaStream_t sf = ctx->side[0];
  if (!full) {
    // (7) Rayleigh-Ritz on C^T C (Gram partials came out of the broadcast pass), rotate both factors
    METIS_CUDA_TRY(metis_launch_pdl((reduce_gram_kernel), dim3((unsigned)metis_ceil_div(kp * kp, 32)), dim3(128), (size_t)(0), sf, gram_c, n_cta_c, kp * kp, gram1, nullptr)); METIS_COUNT_LAUNCH();
    METIS_TRY(launch_eig(sf, gram1, k, kp, evals2, evecs2));
    FactorsArgs f{};
    f.w = evecs2; f.ldw = k; f.n_in = k; f.k = k; f.kp = kp;
    f.basis = basis; f.cols = cols; f.right = out->right; f.keys = keys; f.amax_right = amax + 2;
    f.src = coef; f.ld = kp; f.rows = rows; f.evals = evals2; f.left = out->left; f.sigma_out = out->sigma; f.amax_left = amax + 1;
    METIS_TRY(launch_factors(sf, f, n_cta_cols, n_cta_rows));
  }
  METIS_CUDA_TRY(cudaGetLastError());
  // (8) apply the sign convention and quantize the factors (stored transposed: k x rows, k x cols; blocks along the long dimension)
  metis_nvfp4_t lq = out->left_q, rq = out->right_q;
  lq.rows = k; lq.k_len = rows; rq.rows = k; rq.k_len = cols;
  METIS_TRY(metis_launch_quantize_factors(out->left, rows, out->right, cols, k, rounding, seed, amax + 1, amax + 2, &lq, &rq, sf, keys));
  return metis_join(ctx, s, 0);
}
