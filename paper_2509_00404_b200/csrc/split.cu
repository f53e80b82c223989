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
// The j-th sampled row: one row per stratum of g consecutive rows, offset from Philox (g = 0: every row)
struct RowSample { uint32_t g; uint64_t seed; };
__device__ __forceinline__ int sample_row(const RowSample& rs, int j) {
  if (rs.g == 0u) return j;
  const uint4 w = metis_philox((uint32_t)j, 0u, METIS_STREAM_SAMPLING, 0u, (uint32_t)rs.seed, (uint32_t)(rs.seed >> 32));
  return (int)((uint32_t)j * rs.g + w.x % rs.g);
}
// What the later kernels of a decomposition accumulate into, cleared by its first kernel (a memset of its own was a launch in front of
// every decomposition): amax slots, condition flag, sign keys.
__device__ __forceinline__ void clear_accumulators(float* amax, unsigned long long* keys) {
  if (threadIdx.x < 16) amax[threadIdx.x] = 0.0f;
  if (threadIdx.x < 64) keys[threadIdx.x] = 0ull;
}

// the sampled rows as indices (wide chain)
__global__ void sample_rows_kernel(int* __restrict__ idx, int n_s, RowSample rs) {
  metis_pdl_wait_trigger();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n_s) idx[j] = sample_row(rs, j);
}

// ------------------------------------------------------------------------------------------------
// amax|x| not finite: a NaN or an infinity in the operand (amax is kept as an ordered bit pattern, so a NaN ranks above every number).  For a quantizer
// that does not look itself; a split's amax and eigenvalues are looked at by its factor quantizer.
__global__ void amax_status_kernel(const float* __restrict__ amax, uint32_t* dev_status) {
  metis_pdl_wait_trigger();
  if (threadIdx.x == 0 && !(fabsf(*amax) <= 3.0e38f)) atomicOr(dev_status, METIS_DEV_NONFINITE);
}

// ------------------------------------------------------------------------------------------------
// Gram matrices in FP64 on the FP64 tensor cores: positions are taken 64 at a time, converted to FP64 in shared memory (FP32 -> FP64 conversions are a
// slow-rate instruction: once per element), a warp owns up to six lower 8 x 8 tiles of the result.  The CTAs of a cluster add their tiles through
// distributed shared memory in a fixed order, so that the kernel that needs the matrix (one CTA) adds at most GR_PARTS partials as it loads
// them; a reduction of its own behind 64 partials was a launch of 3 - 4 us in the chain.
constexpr int GR_TILE = 64;
constexpr int GR_TPW = 6;                               // tiles per warp: 45 lower tiles at n = 72 over eight warps
constexpr int GR_PARTS = 16, GR_CLUSTER = 8;
struct GramTiles {
  int t_i[GR_TPW], t_j[GR_TPW], tiles;
  double acc[GR_TPW][2][2];                             // even and odd steps: two chains in flight
};
__device__ __forceinline__ void gram_begin(GramTiles& t, int n8) {
  t.tiles = (n8 / 8) * (n8 / 8 + 1) / 2;
#pragma unroll
  for (int u = 0; u < GR_TPW; ++u) {
    metis_small::lower_tile((int)(threadIdx.x >> 5) + 8 * u, t.t_i[u], t.t_j[u]);
    t.acc[u][0][0] = t.acc[u][0][1] = t.acc[u][1][0] = t.acc[u][1][1] = 0.0;
  }
}
// acc += the product of ROWS positions, tile[position][index] (PITCH 4 or 12 mod 16: conflict-free)
template <int ROWS, int PITCH>
__device__ __forceinline__ void gram_add(GramTiles& t, const double* tile) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q4 = lane & 3;
#pragma unroll
  for (int u = 0; u < GR_TPW; ++u) {
    if (warp + 8 * u < t.tiles) {
      const double* pa = tile + q4 * PITCH + 8 * t.t_i[u] + g;
      const double* pb = tile + q4 * PITCH + 8 * t.t_j[u] + g;
#pragma unroll
      for (int kk = 0; kk < ROWS; kk += 8) {
        metis_small::dmma(t.acc[u][0], pa[kk * PITCH], pb[kk * PITCH]);
        metis_small::dmma(t.acc[u][1], pa[(kk + 4) * PITCH], pb[(kk + 4) * PITCH]);
      }
    }
  }
}
// the cluster's sum into out (n x n); gp: shared memory for 64 doubles per tile, written by nobody else meanwhile; by all 256 threads of every CTA
__device__ __forceinline__ void gram_end(const GramTiles& t, double* gp, int n, double* __restrict__ out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q4 = lane & 3;
#pragma unroll
  for (int u = 0; u < GR_TPW; ++u)
    if (warp + 8 * u < t.tiles)
      *reinterpret_cast<double2*>(gp + 64 * (warp + 8 * u) + 8 * g + 2 * q4) = make_double2(t.acc[u][0][0] + t.acc[u][1][0], t.acc[u][0][1] + t.acc[u][1][1]);
  const uint32_t csize = metis_cluster_size(), rank = metis_cluster_rank(), src = (uint32_t)__cvta_generic_to_shared(gp);
  __syncthreads();
  metis_cluster_sync();
  for (int o = 4 * (int)rank + (tid >> 6); o < t.tiles; o += 4 * (int)csize) {     // four tiles at a time, an entry per thread
    const int e = tid & 63;
    double v[GR_CLUSTER], x = 0.0;
#pragma unroll
    for (uint32_t c = 0; c < GR_CLUSTER; ++c) {
      v[c] = 0.0;
      if (c < csize) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[c]) : "r"(metis_map_to_rank(src + (uint32_t)(64 * o + e) * 8u, c)));
    }
#pragma unroll
    for (uint32_t c = 0; c < GR_CLUSTER; ++c) x += v[c];
    int ti, tj;
    metis_small::lower_tile(o, ti, tj);
    const int i = 8 * ti + (e >> 3), j = 8 * tj + (e & 7);
    if (i < n && j < n) {
      out[i * n + j] = x;
      if (ti != tj) out[j * n + i] = x;
    }
  }
  metis_cluster_sync();                                 // the others may still be reading
}
// the sum of `parts` partials of an entry (at most GR_PARTS), loads in flight
__device__ __forceinline__ double sum_parts(const double* __restrict__ in, int parts, int64_t stride) {
  double a = 0.0;
#pragma unroll
  for (int p0 = 0; p0 < GR_PARTS; p0 += 8) {
    if (p0 >= parts) break;
    double v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = p0 + u < parts ? in[(int64_t)(p0 + u) * stride] : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) a += v[u];
  }
  return a;
}
// cluster and grid of a Gram kernel over `tiles` tiles of positions: at most GR_PARTS clusters, a CTA takes every grid-th tile
inline void gram_grid(int64_t tiles, int* ctas, int* csize) {
  int c = 1;
  while (c < GR_CLUSTER && c < tiles) c *= 2;
  const int64_t n = (tiles + c - 1) / c;
  *csize = c; *ctas = (int)(n < GR_PARTS ? n : GR_PARTS) * c;
}

// Sums column slices of a tensor-core pass in a fixed order, v[position][i] = sum over s of part[s][position][i] (rows `width` wide, i < q), stores them
// row by row (TRANS = 0: out[position][i]) or vector by vector (TRANS = 1: out[i][position]) and forms the Gram matrix of the q vectors.
// out may be null (the slices are then the vectors themselves).
// SOME: of rows that are wider than the q vectors take, only these are read.  For CTAs of several tiles, which are bound by their bytes (every row of 2^20 x 64,
// q = 8 of 48 columns: split 1633 -> 1271 us; 16384 x 4096 at q = 40 of 48: step of the k / v projection 677 -> 669); a CTA of one tile takes half a us longer so.
constexpr size_t SG_SMEM = sizeof(double) * (GR_TILE * LP + 64 * 45);
template <bool TRANS, bool SOME>
__global__ void __launch_bounds__(256)
sum_gram_kernel(const float* __restrict__ part, int slices, int64_t n_pos, int width, int q, float* __restrict__ out, double* __restrict__ gram_part,
                const int* __restrict__ skip) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;                 // second CholeskyQR pass not needed (see chol_kernel)
  extern __shared__ __align__(16) double sg_sm[];
  double *tile = sg_sm, *gp = sg_sm + GR_TILE * LP;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n8 = (q + 7) & ~7;
  GramTiles t;
  gram_begin(t, n8);
  const int64_t tiles = (n_pos + GR_TILE - 1) / GR_TILE;
  for (int64_t ti = blockIdx.x; ti < tiles; ti += gridDim.x) {
    const int64_t p0 = ti * GR_TILE;
    if ((width & 3) == 0) {
      // the tile is one run of 64 * width floats per slice: groups of four, two groups' slices in flight (columns from q on are zeros)
      const int w4 = width >> 2, n4 = SOME ? n8 >> 2 : w4, n_o = (int)min((int64_t)GR_TILE, n_pos - p0) * n4;
      const float4* src = reinterpret_cast<const float4*>(part) + p0 * w4;
      const int64_t stride = n_pos * w4;
      auto place = [&](int o) { return SOME ? o + o / n4 * (w4 - n4) : o; };
      for (int o0 = tid; o0 < GR_TILE * n4; o0 += 512) {
        float4 v[2][8];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int sl = 0; sl < 8; ++sl) v[u][sl] = sl < slices && o0 + 256 * u < n_o ? src[sl * stride + place(o0 + 256 * u)] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int o = o0 + 256 * u, p = o / n4, j = 4 * (o - p * n4);
          if (o >= GR_TILE * n4) break;
          float4 x = v[u][0];
#pragma unroll
          for (int sl = 1; sl < 8; ++sl) { x.x += v[u][sl].x; x.y += v[u][sl].y; x.z += v[u][sl].z; x.w += v[u][sl].w; }
          for (int sl = 8; sl < slices && o < n_o; ++sl) { const float4 y = src[sl * stride + place(o)]; x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w; }
          if (j < n8) {
            *reinterpret_cast<double2*>(tile + p * LP + j) = make_double2((double)x.x, (double)x.y);
            *reinterpret_cast<double2*>(tile + p * LP + j + 2) = make_double2((double)x.z, (double)x.w);
          }
          if (!TRANS && out != nullptr && o < n_o) {
            float* dst = out + (p0 + p) * q + j;
            if ((q & 3) == 0) { if (j < q) *reinterpret_cast<float4*>(dst) = x; }
            else {
              const float e[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
              for (int k = 0; k < 4; ++k) if (j + k < q) dst[k] = e[k];
            }
          }
        }
      }
    } else {
      for (int o = tid; o < GR_TILE * n8; o += 256) {
        const int p = o / n8, j = o - p * n8;
        float x = 0.0f;
        if (p0 + p < n_pos && j < q) {
          for (int sl = 0; sl < slices; ++sl) x += part[(sl * n_pos + p0 + p) * width + j];
          if (!TRANS && out != nullptr) out[(p0 + p) * q + j] = x;
        }
        tile[p * LP + j] = (double)x;
      }
    }
    __syncthreads();
    if (TRANS)
      for (int i = warp; i < q; i += 8)
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (p0 + lane + 32 * h < n_pos) out[(int64_t)i * n_pos + p0 + lane + 32 * h] = (float)tile[(lane + 32 * h) * LP + i];
    gram_add<GR_TILE, LP>(t, tile);
    __syncthreads();
  }
  gram_end(t, gp, q, gram_part + (int64_t)(blockIdx.x / metis_cluster_size()) * q * q);
}

// ------------------------------------------------------------------------------------------------
// largest diagonal entry of a Gram matrix, to 20 bits from below (the high words order like the values); every warp by itself
__device__ __forceinline__ double gram_scale(const double* L, int q) {
  int top = 0;
  for (int i = threadIdx.x & 31; i < q; i += 32) top = max(top, __double2hiint(L[i * LP + i]));
  return __hiloint2double(__reduce_max_sync(0xFFFFFFFFu, top), 0);
}

// H = Z L^-T for eight rows by one warp, in registers: block column b is (Z_b - sum_k H_k L_bk^T) X_b^T with X_b the inverse of the factor's
// 8 x 8 diagonal block.  h: accumulator tiles (lane: row lane / 4, columns 2 (lane % 4) and the next); a tile is the left operand of the next
// product as it stands, its columns taken in the order 2 q, then 2 q + 1.
template <int KT>
__device__ __forceinline__ void solve_rows(double (&h)[KT][2], const double* L, const double (*Xd)[64]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q4 = lane & 3;
#pragma unroll
  for (int b = 0; b < KT; ++b) {
    double acc2[2] = {0.0, 0.0};
#pragma unroll
    for (int k = 0; k < b; ++k) {
      const double2 l = *reinterpret_cast<const double2*>(L + (8 * b + g) * LP + 8 * k + 2 * q4);
      metis_small::dmma(h[b], -h[k][0], l.x);
      metis_small::dmma(acc2, -h[k][1], l.y);
    }
    const double2 x = *reinterpret_cast<const double2*>(Xd[b] + 8 * g + 2 * q4);
    const double a0 = h[b][0] + acc2[0], a1 = h[b][1] + acc2[1];
    h[b][0] = h[b][1] = 0.0;
    metis_small::dmma(h[b], a0, x.x);
    metis_small::dmma(h[b], a1, x.y);
  }
}
// Stores eight rows of H: FP32 rows of z, and the three-term BF16 splits, transposed (hsp[term][vector][row]: pairs of neighbouring rows, an even
// row's lane keeps column j, an odd row's column j + 1).  r: this lane's row.
template <int KT>
__device__ __forceinline__ void store_rows(const double (&h)[KT][2], int64_t r, int64_t n_rows, int q, float* __restrict__ z, __nv_bfloat16* __restrict__ hsp, int jp, int64_t ldh) {
  const int lane = threadIdx.x & 31, q4 = lane & 3;
  const bool odd = lane & 4, in = r < n_rows;
#pragma unroll
  for (int b = 0; b < KT; ++b) {
    const int j = 8 * b + 2 * q4;
    const float v0 = in ? (float)h[b][0] : 0.0f, v1 = in ? (float)h[b][1] : 0.0f;
    if (in) {
      if ((q & 1) == 0) { if (j < q) *reinterpret_cast<float2*>(z + r * q + j) = make_float2(v0, v1); }
      else { if (j < q) z[r * q + j] = v0; if (j + 1 < q) z[r * q + j + 1] = v1; }
    }
    const float other = __shfl_xor_sync(0xFFFFFFFFu, odd ? v0 : v1, 4);
    float x = odd ? other : v0, y = odd ? v1 : other;
    __nv_bfloat16* dst = hsp + (int64_t)(j + (odd ? 1 : 0)) * ldh + (r & ~(int64_t)1);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      const __nv_bfloat162 hb = __floats2bfloat162_rn(x, y);
      const uint32_t w = *reinterpret_cast<const uint32_t*>(&hb);
      x -= __uint_as_float(w << 16); y -= __uint_as_float(w & 0xFFFF0000u);
      *reinterpret_cast<uint32_t*>(dst + (int64_t)t * jp * ldh) = w;
    }
  }
}
// One CholeskyQR pass of many rows, step 1 (one CTA): G = L L^T in FP64 from its partials; writes L and the inverses of its 8 x 8 diagonal blocks
// (l_out: MAXQ x LP, then a block's 64 entries each), so that step 2 is a product on many CTAs.  A pivot below 1e-13 of the largest diagonal marks a
// dependent sketch column: the corresponding column of H = Z L^-T becomes zero instead of amplified noise.
constexpr int CHOL_THREADS = 256, L_DOUBLES = MAXQ * LP + 64 * (MAXQ / 8);
__global__ void __launch_bounds__(CHOL_THREADS)
chol_kernel(const double* __restrict__ gm, int parts, int q, double* __restrict__ l_out, const int* __restrict__ skip, int* __restrict__ well_conditioned) {
  metis_pdl_wait();
  if (skip != nullptr && *skip) return;
  __shared__ __align__(16) double L[MAXQ][LP];
  __shared__ double dmin_s, inv_s[MAXQ];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, q8 = (q + 7) & ~7;
  for (int i = warp; i < q8; i += CHOL_THREADS / 32)
    for (int j = lane; j < q8; j += 32) L[i][j] = i < q && j <= i ? sum_parts(gm + i * q + j, parts, (int64_t)q * q) : 0.0;
  __syncthreads();
  const double gmax = gram_scale(&L[0][0], q);
  metis_small::cta_cholesky<LP>(&L[0][0], q, 1e-13 * gmax, inv_s, &dmin_s, CHOL_THREADS);
  // With every pivot above 1e-8 of the largest diagonal the FP64 factorisation leaves Z L^-T orthonormal to
  // ~1e-8 already, below the FP32 rounding of its storage: the caller's second pass is then skipped.
  metis_pdl_trigger();
  if (tid == 0 && well_conditioned != nullptr) *well_conditioned = (dmin_s > 1e-8 * gmax) ? 1 : 0;
  for (int b = warp; b < q8 / 8; b += CHOL_THREADS / 32) metis_small::invert_diagonal_block<LP>(&L[0][0], inv_s, q, b, l_out + MAXQ * LP + 64 * b, 8);
  for (int o = tid; o < q8 * LP / 2; o += CHOL_THREADS) reinterpret_cast<double2*>(l_out)[o] = reinterpret_cast<const double2*>(&L[0][0])[o];
}

// One CholeskyQR pass of many rows, step 2: Z <- Z L^-T in place, 64 rows per CTA, a warp per eight rows, and the splits of the result.  (As a product with
// the explicit inverse from shared memory, with FP64 copies of Z and the inverse: 1570 instructions a warp, 8 us of a chain.  A triangular solve per
// row, one column after the other, took 15 us for 4096 x 40, 47 us for 16384 x 40 and 186 us for 28672 x 72.)
constexpr int OA_ROWS = 64;
template <int KT>                                       // ceil(q / 8)
__global__ void __launch_bounds__(256)
orth_apply_kernel(float* __restrict__ z, int64_t n_rows, int q, const double* __restrict__ l, const int* __restrict__ skip,
                  __nv_bfloat16* __restrict__ hsp, int jp, int64_t ldh) {
  metis_pdl_wait_trigger();
  if (skip != nullptr && *skip) return;
  __shared__ __align__(16) double L[8 * KT][LP];
  __shared__ __align__(16) double Xd[KT][64];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q4 = lane & 3;
  const int64_t r0 = (int64_t)blockIdx.x * OA_ROWS, r = r0 + 8 * warp + g;
  double h[KT][2];
#pragma unroll
  for (int b = 0; b < KT; ++b) {
    const int j = 8 * b + 2 * q4;
    float2 v = make_float2(0.0f, 0.0f);
    if (r < n_rows && (q & 1) == 0 && j < q) v = *reinterpret_cast<const float2*>(z + r * q + j);
    else if (r < n_rows && (q & 1) != 0) { if (j < q) v.x = z[r * q + j]; if (j + 1 < q) v.y = z[r * q + j + 1]; }
    h[b][0] = (double)v.x; h[b][1] = (double)v.y;
  }
#pragma unroll 4
  for (int o = tid; o < 8 * KT * LP / 2; o += 256) reinterpret_cast<double2*>(&L[0][0])[o] = reinterpret_cast<const double2*>(l)[o];
  for (int o = tid; o < 64 * KT / 2; o += 256) reinterpret_cast<double2*>(&Xd[0][0])[o] = reinterpret_cast<const double2*>(l + MAXQ * LP)[o];
  __syncthreads();
  solve_rows<KT>(h, &L[0][0], Xd);
  store_rows<KT>(h, r, n_rows, q, z, hsp, jp, ldh);     // (rows up to the next multiple of 64 are zeros of the splits)
  if (jp > 8 * KT && tid < 24 * OA_ROWS / 8)            // vectors beyond 8 KT (eight of each term)
    *reinterpret_cast<uint4*>(hsp + ((int64_t)(tid >> 6) * jp + 8 * KT + (tid & 7)) * ldh + r0 + 8 * ((tid >> 3) & 7)) = make_uint4(0u, 0u, 0u, 0u);
}

// Orthonormalisation of a short sketch (the row-sampled case: a few hundred rows) by one cluster: a CTA takes every eighth group of eight rows - the sum of the
// sketch's partials, its part of G = Z^T Z on the FP64 tensor cores, later its rows of H = Z L^-T - and all of them factorise G, whose sum they
// exchange through distributed shared memory, for themselves.  With a pivot below 1e-8 of the largest diagonal a second pass runs on
// the FP64 rows (above that Z L^-T is orthonormal to ~1e-8 already, below the FP32 rounding of its storage); a pivot below 1e-13 marks a
// dependent column, whose column of H is zero.  In one CTA of sixteen warps 17.7 us at 160 x 40 (sum 4.6 k cycles, Gram matrix 4.4 k,
// factor 10.9 k, H 8.5 k) and 52 us at 288 x 72; now 11.2 us (1.4 k, 1.1 k and 3.1 k for the exchange, 8.4 k, 1.9 k) and 22.6 us.
constexpr int GC_THREADS = 256, GC_CLUSTER = 8;
constexpr int64_t GC_MAX_ROWS = 1024;                   // longer sketches: sum_gram_kernel, chol_kernel, orth_apply_kernel
__host__ __device__ constexpr int gram_chol_pitch(int kt) { return 8 * kt + 4; }        // 4 or 12 mod 16: conflict-free fragment loads
__host__ __device__ constexpr int64_t gram_chol_rows(int64_t n_s) { return (n_s / 8 + GC_CLUSTER - 1) / GC_CLUSTER * 8; }      // of a CTA
__host__ __device__ constexpr size_t gram_chol_smem(int64_t n_s, int kt) {
  return sizeof(double) * (size_t)(8 * kt * LP + 64 * (kt * (kt + 1) / 2) + gram_chol_rows(n_s) * gram_chol_pitch(kt));
}
template <int KT>                                       // ceil(q / 8)
__global__ void __launch_bounds__(GC_THREADS, 1)
gram_chol_kernel(const float* __restrict__ zp, int parts, int width, int n_s, int q, float* __restrict__ z, __nv_bfloat16* __restrict__ hsp, int jp, int64_t ldh) {
  metis_pdl_wait();
  constexpr int Q8 = 8 * KT, ZP = gram_chol_pitch(KT), TILES = KT * (KT + 1) / 2, TPW = (TILES + 7) / 8;
  extern __shared__ __align__(16) double gc_sm[];
  double (*L)[LP] = reinterpret_cast<double (*)[LP]>(gc_sm);                     // [Q8][LP]
  double *gp = gc_sm + Q8 * LP, *zs = gp + 64 * TILES;  // [TILES][64], [own rows][ZP]
  __shared__ __align__(16) double Xd[KT][64];
  __shared__ double dmin_s, inv_s[MAXQ];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q4 = lane & 3;
  const int rank = (int)metis_cluster_rank(), groups = (n_s / 8 - rank + GC_CLUSTER - 1) / GC_CLUSTER;         // own groups of eight rows: rank, rank + 8, ...
  // ---- the sketch: eight columns of a row per thread, all partials in flight ----
  for (int o = tid; o < groups * 8 * KT; o += GC_THREADS) {
    const int lr = o / KT, c0 = 8 * (o - lr * KT), r = 8 * (rank + GC_CLUSTER * (lr >> 3)) + (lr & 7);
    const float* src = zp + (int64_t)r * width + c0;        // (a partial's columns beyond q, if it has them, are zeros)
    const int64_t stride = (int64_t)n_s * width;
    float a[8] = {};
    if ((width & 3) == 0) {                              // whole groups of four
#pragma unroll
      for (int p0 = 0; p0 < GR_PARTS; p0 += 8) {
        if (p0 >= parts) break;
        float4 u[8], v[8];
#pragma unroll
        for (int p = 0; p < 8; ++p) {
          u[p] = v[p] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (p0 + p < parts) {
            u[p] = *reinterpret_cast<const float4*>(src + (p0 + p) * stride);
            if (c0 + 4 < width) v[p] = *reinterpret_cast<const float4*>(src + (p0 + p) * stride + 4);
          }
        }
#pragma unroll
        for (int p = 0; p < 8; ++p) { a[0] += u[p].x; a[1] += u[p].y; a[2] += u[p].z; a[3] += u[p].w; a[4] += v[p].x; a[5] += v[p].y; a[6] += v[p].z; a[7] += v[p].w; }
      }
    } else {
#pragma unroll 4
      for (int p = 0; p < parts; ++p)
#pragma unroll
        for (int e = 0; e < 8; ++e) a[e] += c0 + e < q ? src[p * stride + e] : 0.0f;
    }
#pragma unroll
    for (int e = 0; e < 8; e += 2) *reinterpret_cast<double2*>(zs + lr * ZP + c0 + e) = make_double2((double)a[e], (double)a[e + 1]);
  }
  __syncthreads();
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
    for (int u = 0; u < TPW; ++u) {
      const int o = warp + 8 * u;
      if (o < TILES) {
        int ti, tj;
        metis_small::lower_tile(o, ti, tj);
        double acc[2][2] = {};
        for (int r0 = 0; r0 < 8 * groups; r0 += 8)
#pragma unroll
          for (int h = 0; h < 2; ++h) metis_small::dmma(acc[h], zs[(r0 + 4 * h + q4) * ZP + 8 * ti + g], zs[(r0 + 4 * h + q4) * ZP + 8 * tj + g]);
        *reinterpret_cast<double2*>(gp + 64 * o + 8 * g + 2 * q4) = make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
      }
    }
    __syncthreads();
    metis_cluster_sync();                                // (also: every CTA has finished with its L of the pass before)
    // tile o is summed by CTA o % 8, in the order of the ranks, and handed to all
    for (int o = rank + GC_CLUSTER * (tid >> 6); o < TILES; o += GC_CLUSTER * (GC_THREADS / 64)) {
      const int e = tid & 63;
      int ti, tj;
      metis_small::lower_tile(o, ti, tj);
      const uint32_t src = (uint32_t)__cvta_generic_to_shared(gp + 64 * o + e), dst = (uint32_t)__cvta_generic_to_shared(&L[8 * ti + (e >> 3)][8 * tj + (e & 7)]);
      double v[GC_CLUSTER], x = 0.0;
#pragma unroll
      for (uint32_t c = 0; c < GC_CLUSTER; ++c) asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[c]) : "r"(metis_map_to_rank(src, c)));
#pragma unroll
      for (uint32_t c = 0; c < GC_CLUSTER; ++c) x += v[c];
#pragma unroll
      for (uint32_t c = 0; c < GC_CLUSTER; ++c) asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(metis_map_to_rank(dst, c)), "d"(x) : "memory");
    }
    __syncthreads();
    metis_cluster_sync();
    const double gmax = gram_scale(&L[0][0], q);
    metis_small::cta_cholesky<LP>(&L[0][0], q, 1e-13 * gmax, inv_s, &dmin_s, GC_THREADS);
    metis_pdl_trigger();
    const bool last = pass == 1 || dmin_s > 1e-8 * gmax;
    for (int b = warp; b < KT; b += GC_THREADS / 32) metis_small::invert_diagonal_block<LP>(&L[0][0], inv_s, q, b, Xd[b], 8);
    __syncthreads();
    for (int gr = warp; gr < groups; gr += GC_THREADS / 32) {
      double h[KT][2];
      double* row = zs + (8 * gr + g) * ZP + 2 * q4;
#pragma unroll
      for (int b = 0; b < KT; ++b) { const double2 v = *reinterpret_cast<const double2*>(row + 8 * b); h[b][0] = v.x; h[b][1] = v.y; }
      solve_rows<KT>(h, &L[0][0], Xd);
      if (last) store_rows<KT>(h, 8 * (rank + GC_CLUSTER * gr) + g, n_s, q, z, hsp, jp, ldh);
      else {
#pragma unroll
        for (int b = 0; b < KT; ++b) *reinterpret_cast<double2*>(row + 8 * b) = make_double2(h[b][0], h[b][1]);
      }
    }
    if (last) break;
    __syncthreads();
  }
  // the splits' padding: vectors beyond Q8, rows beyond n_s
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  if (jp > Q8 && tid < 24)
    for (int gr = 0; gr < groups; ++gr) *reinterpret_cast<uint4*>(hsp + ((int64_t)(tid >> 3) * jp + Q8 + (tid & 7)) * ldh + 8 * (rank + GC_CLUSTER * gr)) = zero;
  if (rank * GC_THREADS + tid < 3 * jp)
    for (int64_t r = n_s; r < ldh; r += 8) *reinterpret_cast<uint4*>(hsp + (int64_t)(rank * GC_THREADS + tid) * ldh + r) = zero;
  metis_cluster_sync();                                  // (nobody reads another's shared memory any more)
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

// Sums the column slices of the tensor-core broadcast pass in a fixed order: coef[r][j] = sum_s part[s][r][j], writes the residual
// product's operand a6 and, per cluster of CTAs of 32 rows each, the Gram partial of their rows of C (for Rayleigh-Ritz).
template <int KP>
__global__ void __launch_bounds__(256)
coef_finish_kernel(const float* __restrict__ part, int slices, int64_t rows, float* __restrict__ coef,
                   double* __restrict__ gram_part, __nv_bfloat16* __restrict__ a6, int kx) {
  constexpr int CP = KP + 4;                            // 4 mod 16: conflict-free fragment loads
  __shared__ float cfin[32 * KP];
  __shared__ __align__(16) double cd[32 * CP];          // converted once: FP32 -> FP64 is a slow-rate instruction
  __shared__ __align__(16) double gp[64 * (KP / 8) * (KP / 8 + 1) / 2];
  GramTiles gt;
  gram_begin(gt, KP);
  metis_pdl_wait_trigger();
  const int tid = threadIdx.x;
  const int64_t row0 = (int64_t)blockIdx.x * 32;
#pragma unroll
  for (int u = 0; u < 32 * KP / 256; ++u) {
    const int o = tid + 256 * u;
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
    cd[o / KP * CP + o % KP] = (double)v;
  }
  __syncthreads();
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
  gram_add<32, CP>(gt, cd);
  gram_end(gt, gp, KP, gram_part + (int64_t)(blockIdx.x / metis_cluster_size()) * KP * KP);
}

// ------------------------------------------------------------------------------------------------
// Sketch of sampled rows (mma.sync): zp[part][row][j] = sum over the columns of a cluster's CTAs of x[row of the sample, col] * Omega[col, j].
// One CTA = 256 sampled rows x chunks of `ccols` columns (every gridDim.y-th); Omega's slice is generated per chunk (Philox + quantile table)
// straight into shared memory, transposed to [j][col] BF16 (its values are BF16 by construction, so the products are exact and only
// the FP32 accumulation rounds), the first one before the wait for the kernels in front.  The CTAs of a cluster add their sums through
// distributed shared memory in a fixed order, which leaves at most GR_PARTS partials for the kernel that needs Z (64 of them were added
// by a launch of its own).  A full sketch does not come here: it runs on the tcgen05 kernel of the broadcast pass (omega_rows_kernel +
// metis_launch_coeff_tc in its raw mode).
constexpr int SKM_ROWS = 256, SKM_COLS = 256;
__host__ __device__ constexpr int skm_pitch(int nt) { return 8 * nt + 4; }             // floats, of the sums in shared memory
__host__ __device__ constexpr size_t skm_smem(int nt, int ccols) {
  const size_t om = sizeof(__nv_bfloat16) * nt * 8 * (size_t)(ccols + 8), sums = sizeof(float) * SKM_ROWS * skm_pitch(nt);
  return om > sums ? om : sums;
}
template <int NT>                                      // sketch columns / 8, rounded up
__global__ void __launch_bounds__(256)
sketch_mma_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, RowSample rs, int n_s, int q, uint64_t seed, const __nv_bfloat16* __restrict__ lut,
                  float* __restrict__ zp, int ccols, int chunks, float* __restrict__ amax, unsigned long long* __restrict__ keys) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int ids[SKM_ROWS];
  __nv_bfloat16* om = reinterpret_cast<__nv_bfloat16*>(smem);          // [NT*8][pitch]
  float* sums = reinterpret_cast<float*>(smem);                        // [SKM_ROWS][SP], afterwards
  constexpr int SP = skm_pitch(NT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, pitch = ccols + 8;
  const int row0 = blockIdx.x * SKM_ROWS, rw = warp * 32;  // this CTA's rows, this warp's among them
  ids[tid] = row0 + tid < n_s ? sample_row(rs, row0 + tid) : 0;
  const bool busy = row0 + rw < n_s;
  float acc[2][NT][4];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][n][e] = 0.0f;
  for (int i = tid; i < (8 * NT - q) * pitch; i += 256) om[q * pitch + i] = __float2bfloat16_rn(0.0f);         // vectors beyond q
  bool first = true;
  for (int ch = blockIdx.y; ch < chunks; ch += gridDim.y) {
    const int64_t col0 = (int64_t)ch * ccols;              // ccols <= SKM_COLS columns per chunk
    const int ncols = (int)min((int64_t)ccols, cols - col0);
    const uint64_t e_lo = (uint64_t)col0 * q, e_hi = (uint64_t)(col0 + ncols) * q;
    for (uint64_t blk = (e_lo >> 3) + tid; blk <= ((e_hi - 1) >> 3); blk += 256) {
      const uint4 w = metis_philox_block(blk, seed, METIS_STREAM_OMEGA);
      const int rel = (int)((int64_t)(blk << 3) - (int64_t)e_lo);      // element of the chunk; the first block may begin before it
      int c = rel >= 0 ? rel / q : -1, j = rel - c * q;
      if (rel < 0) { c = -((q - 1 - rel) / q); j = rel - c * q; }
#pragma unroll
      for (uint32_t h = 0; h < 8; ++h) {
        if (c >= 0 && c < ncols) om[j * pitch + c] = lut[metis_u16_of(w, h)];
        if (++j == q) { j = 0; ++c; }
      }
    }
    if (first) {
      metis_pdl_wait_trigger();
      if (blockIdx.x == 0 && blockIdx.y == 0) clear_accumulators(amax, keys);
      first = false;
    }
    __syncthreads();
    if (busy) {
      const bool v0 = row0 + rw + g < n_s, v1 = row0 + rw + g + 8 < n_s, v2 = row0 + rw + g + 16 < n_s, v3 = row0 + rw + g + 24 < n_s;
      const __nv_bfloat16 *p0 = x + (int64_t)ids[rw + g] * cols + col0, *p1 = x + (int64_t)ids[rw + g + 8] * cols + col0;
      const __nv_bfloat16 *p2 = x + (int64_t)ids[rw + g + 16] * cols + col0, *p3 = x + (int64_t)ids[rw + g + 24] * cols + col0;
      for (int k0 = 0; k0 < ncols; k0 += 64) {             // four steps' loads in flight
        uint32_t a[4][2][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int kk = k0 + 16 * u + 2 * t;
          const bool in = k0 + 16 * u < ncols;
          a[u][0][0] = in && v0 ? *reinterpret_cast<const uint32_t*>(p0 + kk) : 0u;
          a[u][0][1] = in && v1 ? *reinterpret_cast<const uint32_t*>(p1 + kk) : 0u;
          a[u][0][2] = in && v0 ? *reinterpret_cast<const uint32_t*>(p0 + kk + 8) : 0u;
          a[u][0][3] = in && v1 ? *reinterpret_cast<const uint32_t*>(p1 + kk + 8) : 0u;
          a[u][1][0] = in && v2 ? *reinterpret_cast<const uint32_t*>(p2 + kk) : 0u;
          a[u][1][1] = in && v3 ? *reinterpret_cast<const uint32_t*>(p3 + kk) : 0u;
          a[u][1][2] = in && v2 ? *reinterpret_cast<const uint32_t*>(p2 + kk + 8) : 0u;
          a[u][1][3] = in && v3 ? *reinterpret_cast<const uint32_t*>(p3 + kk + 8) : 0u;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (k0 + 16 * u >= ncols) break;
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const __nv_bfloat16* bp = om + (n * 8 + g) * pitch + k0 + 16 * u + 2 * t;
            const uint32_t b0 = *reinterpret_cast<const uint32_t*>(bp), b1 = *reinterpret_cast<const uint32_t*>(bp + 8);
            mma_bf16(acc[0][n], a[u][0], b0, b1);
            mma_bf16(acc[1][n], a[u][1], b0, b1);
          }
        }
      }
    }
    __syncthreads();                                       // the next chunk's Omega, or the sums, take its place
  }
  if (first) metis_pdl_wait_trigger();                     // a CTA without columns, at the end of a cluster
  if (busy) {
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        float* dst = sums + (rw + m * 16 + g) * SP + n * 8 + 2 * t;
        *reinterpret_cast<float2*>(dst) = make_float2(acc[m][n][0], acc[m][n][1]);
        *reinterpret_cast<float2*>(dst + 8 * SP) = make_float2(acc[m][n][2], acc[m][n][3]);
      }
  }
  const uint32_t csize = metis_cluster_size(), rank = metis_cluster_rank(), src = (uint32_t)__cvta_generic_to_shared(sums);
  __syncthreads();
  metis_cluster_sync();
  const int nr = min(SKM_ROWS, n_s - row0);
  float* out = zp + (int64_t)(blockIdx.y / csize) * n_s * q;
  for (int o = (int)rank * 256 + tid; o < nr * 2 * NT; o += (int)csize * 256) {  // groups of four entries of a row
    const int r = o / (2 * NT), c = 4 * (o % (2 * NT));
    float4 v[GR_CLUSTER];
#pragma unroll
    for (uint32_t u = 0; u < GR_CLUSTER; ++u) {
      v[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (u < csize)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[u].x), "=f"(v[u].y), "=f"(v[u].z), "=f"(v[u].w)
                     : "r"(metis_map_to_rank(src + (uint32_t)(r * SP + c) * 4u, u)));
    }
#pragma unroll
    for (int u = 1; u < GR_CLUSTER; ++u) { v[0].x += v[u].x; v[0].y += v[u].y; v[0].z += v[u].z; v[0].w += v[u].w; }
    float* dst = out + (int64_t)(row0 + r) * q + c;
    if ((q & 3) == 0) { if (c < q) *reinterpret_cast<float4*>(dst) = v[0]; }
    else {
      const float e[4] = {v[0].x, v[0].y, v[0].z, v[0].w};
#pragma unroll
      for (int u = 0; u < 4; ++u) if (c + u < q) dst[u] = e[u];
    }
  }
  metis_cluster_sync();                                    // the others may still be reading
}

// Full-mode sketch on the tcgen05 path: Omega is written once, transposed and zero-padded to nb rows
// (omt[j][col], BF16: its values are BF16 by construction), and Z = X Omega runs on the same kernel as the
// coefficient pass.  One thread per Philox block of eight consecutive elements e = col * q + j.
__global__ void __launch_bounds__(256)
omega_rows_kernel(int64_t cols, int q, int nb, uint64_t seed, const __nv_bfloat16* __restrict__ lut, __nv_bfloat16* __restrict__ omt, float* __restrict__ amax,
                  unsigned long long* __restrict__ keys) {
  metis_pdl_wait_trigger();
  if (keys != nullptr && blockIdx.x == 0) clear_accumulators(amax, keys);
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

// ------------------------------------------------------------------------------------------------
// Projection of sampled rows, M[j][col] = sum over r of H[r][j] x[row r, col], and the Gram matrix M M^T (mma.sync; the contraction runs over rows of the
// row-major x, so that x tiles are staged in shared memory and read back transposed with ldmatrix; H is fed as three BF16 terms).
// A CTA owns 64 columns and walks all rows in chunks of 64 through a ring of asynchronous copies (x gathered by row; it does not depend on
// the kernels before, so its first chunks are on their way before the wait for them); four warps across the columns, two halves
// of a chunk.  The tensor core truncates its sums: that of the leading terms of 16 rows goes into an FP32 total at once, and what it lost, the same
// products less the sum, is an accumulator of its own with the smaller terms.
// With M whole in the CTA its Gram matrix follows from shared memory (see gram_add).  As FP32 multiply-adds over ten slabs of rows, their sum, a
// Gram kernel and its reduction this was four launches, 21 us at 160 x 4096 with q = 40; now 7.
// PARTS (a long sample, see launch_project_gram): a CTA takes one of gridDim.y parts of the rows for its 64 columns and leaves mp[part][col][16 MT];
// sum_gram_kernel does the rest.  These are many CTAs, so two of them share an SM.
constexpr int PG_COLS = 64, PG_K = 64, PG_XP = PG_COLS + 8, PG_HP = PG_K + 8;
__host__ __device__ constexpr int pg_stages(bool in_parts) { return in_parts ? 3 : 4; }
__host__ __device__ constexpr size_t pg_smem(int mt, bool in_parts) {
  const size_t ring = (size_t)pg_stages(in_parts) * (PG_K * PG_XP * 2 + 3 * mt * 16 * PG_HP * 2), post = sizeof(float) * mt * 16 * (PG_COLS + 4) + (in_parts ? 0 : SG_SMEM);
  return ring > post ? ring : post;
}
template <int MT, bool PARTS>                           // sketch columns / 16, rounded up
__global__ void __launch_bounds__(256, PARTS && MT <= 4 ? 2 : 1)
project_gram_kernel(const __nv_bfloat16* __restrict__ x, int64_t cols, RowSample rs, int n_s, int q, const __nv_bfloat16* __restrict__ hsp, int ldh,
                    float* __restrict__ m, double* __restrict__ gram_part, float* __restrict__ mp) {
  extern __shared__ __align__(16) unsigned char psm[];
  constexpr int PG_STAGES = pg_stages(PARTS);
  constexpr int XS_BYTES = PG_K * PG_XP * 2, HS_BYTES = 3 * MT * 16 * PG_HP * 2, STAGE = XS_BYTES + HS_BYTES, MP = PG_COLS + 4;
  float* Ms = reinterpret_cast<float*>(psm);            // [MT * 16][MP], over the ring, which has been read by then
  double *tile = reinterpret_cast<double*>(psm + sizeof(float) * MT * 16 * MP), *gp = tile + GR_TILE * LP;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(psm);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, wn = warp & 3, kh = warp >> 2, n8 = (q + 7) & ~7;
  const int all_chunks = (n_s + PG_K - 1) / PG_K, chunk0 = PARTS ? all_chunks * (int)blockIdx.y / (int)gridDim.y : 0;
  const int n_chunks = PARTS ? all_chunks * ((int)blockIdx.y + 1) / (int)gridDim.y - chunk0 : all_chunks;       // of this CTA's part of the rows
  const int64_t tiles = (cols + PG_COLS - 1) / PG_COLS;
  __shared__ int ids[256];                              // the first rows of the sample (beyond them each copy works its row out)
  ids[tid] = tid < n_s ? sample_row(rs, tid) : 0;
  auto load_x = [&](int64_t col0, int c) {
    const uint32_t xs = sbase + (uint32_t)(c % PG_STAGES) * STAGE;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int rr = (tid >> 3) + 32 * u, c8 = (tid & 7) * 8, r = (chunk0 + c) * PG_K + rr;
      const bool ok = r < n_s && col0 + c8 + 8 <= cols;
      cp_async16(xs + (uint32_t)(rr * PG_XP + c8) * 2u, ok ? x + (int64_t)(r < 256 ? ids[r] : sample_row(rs, r)) * cols + col0 + c8 : x, ok);
    }
  };
  auto load_h = [&](int c) {
    const uint32_t hs = sbase + (uint32_t)(c % PG_STAGES) * STAGE + XS_BYTES;
    for (int i = tid; i < 3 * MT * 16 * (PG_K / 8); i += 256) {
      const int row = i >> 3, k8 = (i & 7) * 8;          // row = term * MT * 16 + j
      cp_async16(hs + (uint32_t)(row * PG_HP + k8) * 2u, hsp + (int64_t)row * ldh + (chunk0 + c) * PG_K + k8, true);
    }
  };
  GramTiles gt;
  gram_begin(gt, n8);
  __syncthreads();
  bool first = true;
  for (int64_t ti = blockIdx.x; ti < tiles; ti += gridDim.x) {
    const int64_t col0 = ti * PG_COLS;
#pragma unroll
    for (int c = 0; c < PG_STAGES - 1; ++c) if (c < n_chunks) load_x(col0, c);
    if (first) { metis_pdl_wait_trigger(); first = false; }
#pragma unroll
    for (int c = 0; c < PG_STAGES - 1; ++c) {            // (the x copies belong to the first group)
      if (c < n_chunks) load_h(c);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float acc[MT][2][4], total[MT][2][4];
#pragma unroll
    for (int a = 0; a < MT; ++a)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e) total[a][n][e] = 0.0f;
    for (int c = 0; c < n_chunks; ++c) {
      asm volatile("cp.async.wait_group %0;" ::"n"(PG_STAGES - 2) : "memory");
      __syncthreads();                                     // chunk c has landed; everyone is done with chunk c - 1
      if (c + PG_STAGES - 1 < n_chunks) { load_x(col0, c + PG_STAGES - 1); load_h(c + PG_STAGES - 1); }
      asm volatile("cp.async.commit_group;" ::: "memory");
      const uint32_t xs = sbase + (uint32_t)(c % PG_STAGES) * STAGE, hs = xs + XS_BYTES;
#pragma unroll
      for (int k2 = 0; k2 < 2; ++k2) {
        const int ks = 2 * kh + k2;
#pragma unroll
        for (int a = 0; a < MT; ++a)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[a][n][e] = 0.0f;
        uint32_t b[4];
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                     : "r"(xs + (uint32_t)((ks * 16 + (lane & 15)) * PG_XP + wn * 16 + (lane >> 4) * 8) * 2u));
#pragma unroll
        for (int a = 0; a < MT; ++a)
#pragma unroll
          for (int sp = 0; sp < 3; ++sp) {
            uint32_t af[4];
            const uint32_t addr = hs + (uint32_t)(((sp * MT + a) * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * PG_HP + ks * 16 + (lane >> 4) * 8) * 2u;
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(af[0]), "=r"(af[1]), "=r"(af[2]), "=r"(af[3]) : "r"(addr));
            mma_bf16(acc[a][0], af, b[0], b[1]);
            mma_bf16(acc[a][1], af, b[2], b[3]);
            if (sp == 0) {                                 // what the sum lost: the same products less what it kept
#pragma unroll
              for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) { total[a][n][e] += acc[a][n][e]; acc[a][n][e] = -acc[a][n][e]; }
              mma_bf16(acc[a][0], af, b[0], b[1]);
              mma_bf16(acc[a][1], af, b[2], b[3]);
            }
          }
#pragma unroll
        for (int a = 0; a < MT; ++a)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) total[a][n][e] += acc[a][n][e];
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();                                       // the ring has been read
#pragma unroll
    for (int half = 0; half < 2; ++half) {                 // the second half of the chunks is added to the first
      if (kh == half)
#pragma unroll
        for (int a = 0; a < MT; ++a)
#pragma unroll
          for (int n = 0; n < 2; ++n)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float& o = Ms[(a * 16 + g + 8 * (e >> 1)) * MP + wn * 16 + n * 8 + 2 * t + (e & 1)];
              o = half ? o + total[a][n][e] : total[a][n][e];
            }
      __syncthreads();
    }
    if constexpr (PARTS) {                                 // (a tile per CTA)
      for (int o = tid; o < PG_COLS * 4 * MT; o += 256) {
        const int c = o / (4 * MT), j = 4 * (o - c * 4 * MT);
        if (col0 + c < cols)
          *reinterpret_cast<float4*>(mp + ((int64_t)blockIdx.y * cols + col0 + c) * (16 * MT) + j) =
              make_float4(Ms[j * MP + c], Ms[(j + 1) * MP + c], Ms[(j + 2) * MP + c], Ms[(j + 3) * MP + c]);
      }
      return;
    }
    for (int o = tid; o < q * (PG_COLS / 4); o += 256) {
      const int j = o >> 4, c4 = (o & 15) * 4;
      if (col0 + c4 < cols) *reinterpret_cast<float4*>(m + (int64_t)j * cols + col0 + c4) = *reinterpret_cast<const float4*>(Ms + j * MP + c4);
    }
    for (int o = tid; o < n8 * GR_TILE; o += 256) {        // (vectors q ... n8 - 1 and columns beyond the matrix are zeros)
      const int j = o >> 6, c = o & 63;
      tile[c * LP + j] = (double)Ms[j * MP + c];
    }
    __syncthreads();
    gram_add<GR_TILE, LP>(gt, tile);
    __syncthreads();                                       // the next tile's ring lies over it
  }
  if (first) metis_pdl_wait_trigger();                     // a CTA without columns, at the end of a cluster
  gram_end(gt, gp, q, gram_part + (int64_t)(blockIdx.x / metis_cluster_size()) * q * q);
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

// CTAs and cluster of coef_finish_kernel, 32 rows to a CTA, a Gram partial to a cluster
void coef_grid(int64_t rows, int* ctas, int* csize) {
  const int64_t n = metis_ceil_div(rows, 32);
  int c = 1;
  while (c < GR_CLUSTER && c < n) c *= 2;
  *csize = c; *ctas = (int)(metis_ceil_div(n, c) * c);
}
// accumulator columns of the tensor-core sketch: k + p rounded up to what the coefficient kernel is built for
int sketch_tc_cols(int q) { return q <= 48 ? 48 : 96; }

// Column chunks of a sampled sketch: 64 columns each (a 160-row sketch has one row block, so narrow chunks are what gives it CTAs), wider ones or more than
// one to a CTA beyond 128 CTAs, so that the clusters leave at most GR_PARTS partials.
// (of any length of the sample the shortest leaves the most)
struct SketchGrid { int ccols, chunks, ctas, csize, parts; };
SketchGrid sketch_grid(int64_t cols, int64_t n_s) {
  SketchGrid s{};
  s.ccols = cols <= 64 * 128 ? 64 : (cols <= 128 * 128 ? 128 : SKM_COLS);
  // a long sample has its CTAs from its rows: fewer sums to exchange
  while (n_s > GC_MAX_ROWS && s.ccols < SKM_COLS && metis_ceil_div(n_s, SKM_ROWS) * metis_ceil_div(cols, 2 * s.ccols) >= 296) s.ccols *= 2;
  s.chunks = (int)metis_ceil_div(cols, s.ccols);
  gram_grid(s.chunks, &s.ctas, &s.csize);
  s.parts = s.ctas / s.csize;
  return s;
}

struct SplitWs {
  size_t amax, zp, omt, z, gram, gram1, linv, evals, evecs, mp, m, basis, coef, keys, evals2, evecs2, bs,
      gram_c, part, a6, b6, hsp, total;
};

SplitWs split_ws_layout(int64_t rows, int64_t cols, int k, int p, int64_t n_s) {
  SplitWs w{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += (bytes + 255) & ~(size_t)255; return o; };
  const int q = k + p;
  w.amax = take(256);
  // the full-mode tensor-core sketch writes slices x rows x nb partials into the buffer of the sampled one's
  const int nb_sk = sketch_tc_cols(q);
  const size_t zp_mma = (size_t)sketch_grid(cols, 0).parts * n_s * q, zp_tc = (size_t)metis_coeff_slices(rows, cols, nullptr) * rows * nb_sk;
  w.zp = take(sizeof(float) * (zp_mma > zp_tc ? zp_mma : zp_tc));
  w.omt = take(sizeof(__nv_bfloat16) * (size_t)nb_sk * cols);
  w.z = take(sizeof(float) * (size_t)n_s * q);
  w.gram = take(sizeof(double) * GR_PARTS * MAXQ * MAXQ);
  w.linv = take(sizeof(double) * L_DOUBLES);
  w.gram1 = take(sizeof(double) * MAXQ * MAXQ);
  w.evals = take(sizeof(double) * MAXQ);
  w.evecs = take(sizeof(double) * MAXQ * MAXQ);
  w.mp = take(sizeof(float) * (size_t)8 * ((q + 15) / 16 * 16) * cols);                 // tensor-core projection: at most eight slices
  w.m = take(sizeof(float) * (size_t)q * cols);
  w.basis = take(sizeof(float) * (size_t)k * cols);
  const int kp = (k + 15) / 16 * 16;
  w.coef = take(sizeof(float) * (size_t)kp * rows);
  w.part = take(sizeof(float) * (size_t)metis_coeff_slices(rows, cols, nullptr) * kp * rows);
  w.a6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * rows);
  w.b6 = take(sizeof(__nv_bfloat16) * (size_t)metis_residual_kx(kp) * cols);
  w.hsp = take(sizeof(__nv_bfloat16) * 3 * (size_t)((q + 15) / 16 * 16) * (size_t)((n_s + 63) / 64 * 64));
  w.bs = take(sizeof(__nv_bfloat16) * 3 * (size_t)kp * cols);
  int ctas_c, csize_c;
  coef_grid(rows, &ctas_c, &csize_c);
  w.gram_c = take(sizeof(double) * (size_t)(ctas_c / csize_c) * kp * kp);
  w.keys = take(sizeof(unsigned long long) * MAXQ);
  w.evals2 = take(sizeof(double) * MAXQ);
  w.evecs2 = take(sizeof(double) * MAXQ * MAXQ);
  w.total = off;
  return w;
}

metis_status_t launch_eig(cudaStream_t s, const double* g, int parts, int n, int ld, double* evals, double* evecs) {
  const size_t smem = metis_small::eig_smem(n);
#define METIS_EIG(NT8) case NT8: METIS_CUDA_TRY(metis_launch_pdl((metis_small::eig_kernel<NT8>), dim3(1), dim3(metis_small::eig_threads(NT8)), smem, s, g, parts, n, ld, evals, evecs)); break
  switch ((n + 7) / 8) {
    METIS_EIG(1); METIS_EIG(2); METIS_EIG(3); METIS_EIG(4); METIS_EIG(5); METIS_EIG(6); METIS_EIG(7); METIS_EIG(8); METIS_EIG(9);
    default: return METIS_ERR_SHAPE;
  }
#undef METIS_EIG
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

// Gram partials of vectors given as column slices of a tensor-core pass (see sum_gram_kernel); returns the number of partials
template <bool TRANS>
metis_status_t launch_sum_gram(cudaStream_t s, const float* part, int slices, int64_t n_pos, int width, int q, float* out, double* gram, const int* skip, int* parts) {
  int ctas, csize;
  gram_grid(metis_ceil_div(n_pos, GR_TILE), &ctas, &csize);
  *parts = ctas / csize;
  const bool some = metis_ceil_div(n_pos, GR_TILE) > ctas && width % 4 == 0 && (q + 7) / 8 * 8 < width;
  METIS_CUDA_TRY(metis_launch_pdl_cluster(some ? sum_gram_kernel<TRANS, true> : sum_gram_kernel<TRANS, false>, dim3((unsigned)ctas), dim3(256), SG_SMEM, s, 0, csize, part, slices, n_pos,
                                          width, q, out, gram, skip)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}
// M = H^T x of sampled rows and its Gram partials.  A tile's CTA walks all rows; where that is long, up to eight CTAs take a part of the rows each and
// sum_gram_kernel adds the parts (mp).  The rule counts rounds of CTAs times chunks of 64 rows behind one another (1.4 us, a third more with two CTAs on an
// SM), six more for a CTA's start and end and twelve for the launch behind; samples of up to 1024 rows have no use for it.  Whole split, all rows in one CTA -> in
// parts (and as slabs of 512 rows with FP32 partials, before both): p = 8, 8192 of 16384 x 1024, k = 32 355 -> 201 us (230); 4096 of 16384 x 4096 341 -> 269
// (282); every row of 16384 x 4096 in a sample, k = 64 1247 -> 816 (881); 1312 of 131072 x 256, k = 8 171 -> 153 (270); 8192 of 16384 x 14336 1030 -> 830 (797).
metis_status_t launch_project_gram(metis_context* ctx, cudaStream_t s, const __nv_bfloat16* x, int64_t cols, const RowSample& rs, int n_s, int q, const __nv_bfloat16* hsp, int ldh, float* m, double* gram,
                                   float* mp, int* parts) {
  const int64_t tiles = metis_ceil_div(cols, PG_COLS), chunks = metis_ceil_div(n_s, PG_K);
  int ctas, csize, slices = 1;
  gram_grid(tiles, &ctas, &csize);
  const bool two = q <= 64;                             // CTAs on an SM
  int64_t best = (chunks + 6) * metis_ceil_div(tiles, ctas < 120 ? ctas : 120) * 3;                  // (fifteen clusters of eight are resident)
  for (int n = 2; n <= 8 && chunks > 16; ++n) {
    const int64_t load = tiles * n, sms = ctx->sm_count, rounds = load <= sms || !two ? 3 * metis_ceil_div(load, sms) : 4 * metis_ceil_div(load, 2 * sms);
    const int64_t cost = (metis_ceil_div(chunks, n) + 6) * rounds + 36;
    if (cost < best) { best = cost; slices = n; }
  }
  *parts = ctas / csize;
#define METIS_PG(MT) case MT: \
    if (slices > 1) METIS_CUDA_TRY(metis_launch_pdl(project_gram_kernel<MT, true>, dim3((unsigned)tiles, (unsigned)slices), dim3(256), pg_smem(MT, true), s, x, cols, rs, n_s, q, hsp, ldh, m, gram, mp)); \
    else METIS_CUDA_TRY(metis_launch_pdl_cluster(project_gram_kernel<MT, false>, dim3((unsigned)ctas), dim3(256), pg_smem(MT, false), s, 0, csize, x, cols, rs, n_s, q, hsp, ldh, m, gram, (float*)nullptr)); \
    break
  switch ((q + 15) / 16) {
    METIS_PG(1); METIS_PG(2); METIS_PG(3); METIS_PG(4); METIS_PG(5);
    default: return METIS_ERR_SHAPE;
  }
#undef METIS_PG
  METIS_COUNT_LAUNCH();
  return slices > 1 ? launch_sum_gram<true>(s, mp, slices, cols, (q + 15) / 16 * 16, q, m, gram, nullptr, parts) : METIS_OK;
}
metis_status_t launch_sketch(cudaStream_t s, const SketchGrid& sk, const __nv_bfloat16* x, int64_t cols, const RowSample& rs, int n_s, int q, uint64_t seed, const __nv_bfloat16* lut, float* zp,
                             float* amax, unsigned long long* keys) {
  const dim3 grid((unsigned)metis_ceil_div(n_s, SKM_ROWS), (unsigned)sk.ctas);
#define METIS_SK(NT) case NT: METIS_CUDA_TRY(metis_launch_pdl_cluster(sketch_mma_kernel<NT>, grid, dim3(256), skm_smem(NT, sk.ccols), s, 1, sk.csize, x, cols, rs, n_s, q, seed, lut, zp, \
                                                                       sk.ccols, sk.chunks, amax, keys)); break
  switch ((q + 7) / 8) {
    METIS_SK(1); METIS_SK(2); METIS_SK(3); METIS_SK(4); METIS_SK(5); METIS_SK(6); METIS_SK(7); METIS_SK(8); METIS_SK(9);
    default: return METIS_ERR_SHAPE;
  }
#undef METIS_SK
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}
metis_status_t launch_gram_chol(cudaStream_t s, const float* zp, int parts, int width, int n_s, int q, float* z, __nv_bfloat16* hsp, int jp, int64_t ldh) {
#define METIS_GC(KT) case KT: METIS_CUDA_TRY(metis_launch_pdl_cluster(gram_chol_kernel<KT>, dim3(GC_CLUSTER), dim3(GC_THREADS), gram_chol_smem(n_s, KT), s, 0, GC_CLUSTER, zp, parts, width, n_s, q, z, hsp, jp, ldh)); break
  switch ((q + 7) / 8) {
    METIS_GC(1); METIS_GC(2); METIS_GC(3); METIS_GC(4); METIS_GC(5); METIS_GC(6); METIS_GC(7); METIS_GC(8); METIS_GC(9);
    default: return METIS_ERR_SHAPE;
  }
#undef METIS_GC
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

metis_status_t launch_orth_apply(cudaStream_t s, float* z, int64_t n_s, int q, const double* linvt, const int* skip, __nv_bfloat16* hsp, int jp, int64_t ldh) {
  const dim3 grid((unsigned)metis_ceil_div(n_s, OA_ROWS));
#define METIS_OA(KT) METIS_CUDA_TRY(metis_launch_pdl((orth_apply_kernel<KT>), grid, dim3(256), (size_t)0, s, z, n_s, q, linvt, skip, hsp, jp, ldh)); break
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
  if (n <= MAXQ) return launch_eig(s, gram1, 1, n, n, evals, evecs);               // a small rank with a large oversampling
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
    METIS_CUDA_TRY(metis_launch_pdl((sample_rows_kernel), dim3((unsigned)metis_ceil_div(n_s, 256)), dim3(256), (size_t)(0), s, idx, (int)n_s,
                                    RowSample{(uint32_t)(rows / n_s), seed})); METIS_COUNT_LAUNCH();
    METIS_CUDA_TRY(metis_launch_pdl(metis_wide::gather_rows_kernel, dim3((unsigned)metis_ceil_div(n_s * (cols / 8), 256)), dim3(256), (size_t)0, s, x, cols,
                                    (const int*)idx, (int)n_s, xs)); METIS_COUNT_LAUNCH();
    xr = xs;
  }
  // (2) sketch Z = xr Omega on the tensor cores, WIDE_SK sketch columns per launch
  const int nbq = (q + WIDE_SK - 1) / WIDE_SK * WIDE_SK;
  {
    const uint64_t blocks = ((uint64_t)cols * q + 7) / 8;
    METIS_CUDA_TRY(metis_launch_pdl((omega_rows_kernel), dim3((unsigned)metis_ceil_div((int64_t)blocks, 256)), dim3(256), (size_t)(0), s, cols, q, nbq, seed, ctx->quantile_lut, omt,
                                    (float*)nullptr, (unsigned long long*)nullptr)); METIS_COUNT_LAUNCH();
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
  METIS_CUDA_TRY(cudaGetLastError());
  const metis_split_checks checks{amax, evals, k, ctx->dev_status};
  metis_nvfp4_t lq = out->left_q, rq = out->right_q;
  lq.rows = k; lq.k_len = rows; rq.rows = k; rq.k_len = cols;
  METIS_TRY(metis_launch_quantize_factors(out->left, rows, out->right, cols, k, rounding, seed, amax + 1, amax + 2, &lq, &rq, sf, nullptr, &checks));
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
#define METIS_FR_ATTR(KT) METIS_CUDA_TRY(cudaFuncSetAttribute(basis_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fr_smem(MAXQ))); \
  METIS_CUDA_TRY(cudaFuncSetAttribute(factors_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fr_smem(MAXQ)))
  METIS_FR_ATTR(1); METIS_FR_ATTR(2); METIS_FR_ATTR(3); METIS_FR_ATTR(4); METIS_FR_ATTR(5); METIS_FR_ATTR(6); METIS_FR_ATTR(7); METIS_FR_ATTR(8);
#undef METIS_FR_ATTR
#define METIS_EIG_ATTR(NT8) METIS_CUDA_TRY(cudaFuncSetAttribute(metis_small::eig_kernel<NT8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)metis_small::eig_smem(8 * NT8)))
  METIS_EIG_ATTR(1); METIS_EIG_ATTR(2); METIS_EIG_ATTR(3); METIS_EIG_ATTR(4); METIS_EIG_ATTR(5); METIS_EIG_ATTR(6); METIS_EIG_ATTR(7); METIS_EIG_ATTR(8); METIS_EIG_ATTR(9);
#undef METIS_EIG_ATTR
#define METIS_GC_ATTR(KT) METIS_CUDA_TRY(cudaFuncSetAttribute(gram_chol_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gram_chol_smem(GC_MAX_ROWS, KT))); \
  METIS_CUDA_TRY(cudaFuncSetAttribute(sketch_mma_kernel<KT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)skm_smem(KT, SKM_COLS)))
  METIS_GC_ATTR(1); METIS_GC_ATTR(2); METIS_GC_ATTR(3); METIS_GC_ATTR(4); METIS_GC_ATTR(5); METIS_GC_ATTR(6); METIS_GC_ATTR(7); METIS_GC_ATTR(8); METIS_GC_ATTR(9);
#undef METIS_GC_ATTR
#define METIS_SG_ATTR(T, S) METIS_CUDA_TRY(cudaFuncSetAttribute(sum_gram_kernel<T, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SG_SMEM))
  METIS_SG_ATTR(false, false); METIS_SG_ATTR(false, true); METIS_SG_ATTR(true, false); METIS_SG_ATTR(true, true);
#undef METIS_SG_ATTR
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
#define METIS_PP_ATTR(MT) METIS_CUDA_TRY(cudaFuncSetAttribute(project_gram_kernel<MT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pg_smem(MT, false))); \
  METIS_CUDA_TRY(cudaFuncSetAttribute(project_gram_kernel<MT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pg_smem(MT, true)))
  METIS_PP_ATTR(1); METIS_PP_ATTR(2); METIS_PP_ATTR(3); METIS_PP_ATTR(4); METIS_PP_ATTR(5);
#undef METIS_PP_ATTR
  return METIS_OK;
}

// flags METIS_DEV_NONFINITE when *amax (the amax of a tensor about to be quantized) is not a finite number
metis_status_t metis_launch_amax_check(metis_context* ctx, const float* amax, cudaStream_t s) {
  METIS_CUDA_TRY(metis_launch_pdl(amax_status_kernel, dim3(1), dim3(32), (size_t)0, s, amax, ctx->dev_status));
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
  // every buffer grows with the sample count: the FULL sketch (n_s = rows) bounds every other case
  return split_ws_layout(rows, cols, k, p, rows).total;
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
  // (1) row sample and (2) sketch on the tensor cores; the first kernel also clears the amax slots of x, left and right, the condition flag and the
  // sign keys.  amax|x| for the residual's tensor scale: fused into the sketch pass (FULL) or the broadcast pass (SAMPLED).
  const RowSample rs{full ? 0u : (uint32_t)(rows / n_s), seed};
  __nv_bfloat16* omt = reinterpret_cast<__nv_bfloat16*>(wsb + L.omt);
  const int nb_sk = sketch_tc_cols(q), jp = (q + 15) / 16 * 16, ldh = (int)((n_s + 63) / 64 * 64);
  const bool one_cluster = n_s <= GC_MAX_ROWS;
  int parts = 0, slices_z = 0, width_z = q;             // the sketch's partials: zp[slices_z][n_s][width_z]
  if (full) {
    const uint64_t blocks = ((uint64_t)cols * q + 7) / 8;
    METIS_CUDA_TRY(metis_launch_pdl((omega_rows_kernel), dim3((unsigned)metis_ceil_div((int64_t)blocks, 256)), dim3(256), (size_t)(0), s, cols, q, nb_sk, seed, ctx->quantile_lut, omt,
                                    amax, keys)); METIS_COUNT_LAUNCH();
    if (src_amax != nullptr) METIS_CUDA_TRY(cudaMemcpyAsync(amax, src_amax, sizeof(float), cudaMemcpyDeviceToDevice, s));
    METIS_TRY(metis_launch_coeff_tc(ctx, x, rows, cols, omt, nb_sk / 3, zp, amax, 1, s));
    slices_z = metis_coeff_slices(rows, cols, nullptr); width_z = nb_sk;
  } else {
    const SketchGrid sk = sketch_grid(cols, n_s);
    METIS_TRY(launch_sketch(s, sk, x, cols, rs, (int)n_s, q, seed, ctx->quantile_lut, zp, amax, keys));
    if (src_amax != nullptr) METIS_CUDA_TRY(cudaMemcpyAsync(amax, src_amax, sizeof(float), cudaMemcpyDeviceToDevice, s));
    slices_z = sk.parts;
  }
  // (3) CholeskyQR2: orthonormal basis H of range(Z), its BF16 splits for the projection
  if (one_cluster) {
    METIS_TRY(launch_gram_chol(s, zp, slices_z, width_z, (int)n_s, q, z, hsp, jp, ldh));
  } else {
    for (int pass = 0; pass < 2; ++pass) {
      const int* skip = pass == 0 ? nullptr : cond_flag;
      if (pass == 0) METIS_TRY(launch_sum_gram<false>(s, zp, slices_z, n_s, width_z, q, z, gram, skip, &parts));
      else METIS_TRY(launch_sum_gram<false>(s, z, 1, n_s, q, q, nullptr, gram, skip, &parts));
      METIS_CUDA_TRY(metis_launch_pdl((chol_kernel), dim3(1), dim3(CHOL_THREADS), (size_t)0, s, (const double*)gram, parts, q, linvt, skip, pass == 0 ? cond_flag : (int*)nullptr)); METIS_COUNT_LAUNCH();
      METIS_TRY(launch_orth_apply(s, z, n_s, q, linvt, skip, hsp, jp, ldh));
    }
  }
  // (4) M = H^T x[S,:] and M M^T, eigen-decomposition, right basis
  if (full && n_s >= 1024 && metis_project_tc_usable(x, hsp, cols, jp)) {
    // every row, in order: M^T = x^T H on the tcgen05 kernel of the broadcast pass (x as an MN-major operand)
    METIS_TRY(metis_launch_project_tc(ctx, x, rows, cols, hsp, jp, ldh, mp, s));
    METIS_TRY(launch_sum_gram<true>(s, mp, metis_project_slices(rows, cols), cols, jp, q, m, gram, nullptr, &parts));
  } else {
    METIS_TRY(launch_project_gram(ctx, s, x, cols, rs, (int)n_s, q, hsp, ldh, m, gram, mp, &parts));
  }
  METIS_TRY(launch_eig(s, gram, parts, q, q, evals, evecs));
  // (5) right basis and its splits; coefficients of every row in the basis, (6) fused residual + quantizer
  int ctas_c, csize_c;                                    // of the coefficients' last kernel
  coef_grid(rows, &ctas_c, &csize_c);
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
#define METIS_CF(KP) METIS_CUDA_TRY(metis_launch_pdl_cluster((coef_finish_kernel<KP>), dim3((unsigned)ctas_c), dim3(256), (size_t)(0), s, 0, csize_c, (const float*)part, slices, rows, coef, gram_c, a6, kx6)); break
    switch (kp) {
      case 16: METIS_CF(16);
      case 32: METIS_CF(32);
      case 48: METIS_CF(48);
      default: METIS_CF(64);
    }
#undef METIS_CF
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
  }
  cudaStream_t sf = ctx->side[0];
  if (!full) {
    // (7) Rayleigh-Ritz on C^T C (Gram partials came out of the broadcast pass), rotate both factors
    int parts_c = ctas_c / csize_c;
    const double* g2 = gram_c;
    if (parts_c > GR_PARTS) {                             // more than 4096 rows: summed on many CTAs first
      METIS_CUDA_TRY(metis_launch_pdl((reduce_gram_kernel), dim3((unsigned)metis_ceil_div(kp * kp, 32)), dim3(128), (size_t)(0), sf, (const double*)gram_c, parts_c, kp * kp, gram1, (const int*)nullptr)); METIS_COUNT_LAUNCH();
      g2 = gram1; parts_c = 1;
    }
    METIS_TRY(launch_eig(sf, g2, parts_c, k, kp, evals2, evecs2));
    FactorsArgs f{};
    f.w = evecs2; f.ldw = k; f.n_in = k; f.k = k; f.kp = kp;
    f.basis = basis; f.cols = cols; f.right = out->right; f.keys = keys; f.amax_right = amax + 2;
    f.src = coef; f.ld = kp; f.rows = rows; f.evals = evals2; f.left = out->left; f.sigma_out = out->sigma; f.amax_left = amax + 1;
    METIS_TRY(launch_factors(sf, f, n_cta_cols, n_cta_rows));
  }
  METIS_CUDA_TRY(cudaGetLastError());
  // (8) apply the sign convention and quantize the factors (stored transposed: k x rows, k x cols; blocks along the long dimension), status of the split
  metis_nvfp4_t lq = out->left_q, rq = out->right_q;
  lq.rows = k; lq.k_len = rows; rq.rows = k; rq.k_len = cols;
  const metis_split_checks checks{amax, evals, k, ctx->dev_status};
  METIS_TRY(metis_launch_quantize_factors(out->left, rows, out->right, cols, k, rounding, seed, amax + 1, amax + 2, &lq, &rq, sf, keys, &checks));
  return metis_join(ctx, s, 0);
}
