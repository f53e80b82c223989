// Split-FP4 linear layer: forward (Eq. 2), input gradient (Eq. 3) and weight gradient (Section 3.2).
//
// With both operands written as  Ta = Fo_a diag(sa) Fc_a^T + Res_a  (M x K) and
// Tb = Fo_b diag(sb) Fc_b^T + Res_b (N x K), where Fc_* are the factors lying along the contraction
// axis and Fo_* those lying along the output axes, the product expands into
//
//   Ta Tb^T = Res_a Res_b^T                          main FP4 GEMM           (M x N)
//           + (G1 + Fo_a sa P) sb Fo_b^T             G1 = Res_a Fc_b (M x kb), P = Fc_a^T Fc_b (ka x kb)
//           + (Fo_a sa) Wt^T                         Wt = Res_b Fc_a (N x ka)
//
// i.e. one large and three skinny block-scaled FP4 GEMMs followed by a rank-(ka+kb) FP32 update.
// All four quantized cross terms of the paper's expansion are kept.
#include "common.cuh"

#include <cuda_fp16.h>

bool metis_gemm_tc_can_fuse(const metis_nvfp4_t* a, const metis_nvfp4_t* b);
metis_status_t metis_launch_gemm_tc_fused(metis_context* ctx, const metis_nvfp4_t* a, const metis_nvfp4_t* b, void* d,
                                          int d_dtype, int64_t ldd, const void* lx, const void* rx, int kx, cudaStream_t s);

namespace {

__device__ __forceinline__ float deq_at(const uint8_t* codes, const uint8_t* sf, int layout, int64_t k_len, int64_t r,
                                        int64_t c) {
  const uint32_t byte = codes[r * (k_len / 2) + c / 2];
  const uint32_t code = (c & 1) ? (byte >> 4) : (byte & 15u);
  return metis_e2m1_value(code) * metis_e4m3_value(sf[metis_sf_offset(r, c / 16, k_len / 16, layout)]);
}

// Finishes the two skinny operands of the rank-(ka+kb) update.  Layout: Lcat [M][kb + ka], Rcat [N][kb + ka].  On entry Lcat[:, :kb] holds
// G1 and Rcat[:, kb:] holds Wt (written there by the skinny GEMMs).  With A = (G1 + Fo_a sa P) sb the result is
//   lx == nullptr:  in place, Lcat = [A | Fo_a sa], Rcat = [Fo_b | Wt]
//   else:           the BF16 operands of the in-accumulator correction, zero padded to kx columns.  A dequantized factor entry is an
//                   E2M1 x E4M3 product (six significant bits): with its FP32 scales moved to the other operand it is exact in BF16
//                   and needs no low part, so each of the two rank-k terms costs two column groups instead of three:
//                     Lx = [ A' hi | A' lo | Fa | Fa ],  A' = A ts_b / alpha        (k_b columns), Fa = Fo_a / ts_a (k_a)
//                     Rx = [ Fb   | Fb   | B hi | B lo ],  Fb = Fo_b / ts_b (k_b),  B = Wt sa ts_a / alpha          (k_a columns)
// A warp takes R rows (lane: vectors lane and lane + 32): every global load is issued before the first value is used, and a row of P in shared memory serves R rows.
// Latency is what it costs (some 1.6 k instructions of a warp at nine cycles each with R = 4, J = 2 and two warps to a scheduler: 13 us for 4096 rows), so R is 1
// until every scheduler has some eight warps, and ranks up to 32 have an instance of their own.  One row per warp for any number of rows, the finished rows
// through shared memory and FP32 operands written beside the BF16 ones: 17.8 us for 16384 + 4096 rows at k = 32, 8 for 4096; now 9 - 10 and 6.
// the two E2M1 codes of the low byte as FP16 (exact)
__device__ __forceinline__ __half2 e2m1x2_to_half2(uint32_t byte) {
  uint32_t w;
  asm("{ .reg .b8 t; cvt.u8.u32 t, %1; cvt.rn.f16x2.e2m1x2 %0, t; }" : "=r"(w) : "r"(byte));
  return *reinterpret_cast<const __half2*>(&w);
}
struct FinishArgs {
  int64_t M, N;
  int ka, kb, kx, foa_layout, fob_layout;
  const uint8_t *foa_codes, *foa_sf, *fob_codes, *fob_sf;
  const float *foa_ts, *sa, *fob_ts, *sb, *pm;
  float *lcat, *rcat;
  __nv_bfloat16 *lx, *rx;
  const float *res_a_ts, *res_b_ts;
};
// Two products' operands in one launch: blocks below n_first belong to the first.
template <int R, int J>                                     // rows per warp: 1, 2 or 4; 32-vector groups of the ranks: 1 or 2
__global__ void __launch_bounds__(256, J == 1 ? (R == 1 ? 6 : (R == 2 ? 5 : 4)) : (R == 4 ? 3 : 4))          // one wave where the rows allow it
lowrank_finish_kernel(const __grid_constant__ FinishArgs first, const __grid_constant__ FinishArgs second, int n_first) {
  const bool is_first = (int)blockIdx.x < n_first;
  const FinishArgs& f = is_first ? first : second;
  const int64_t M = f.M, N = f.N;
  const int ka = f.ka, kb = f.kb, kx = f.kx, foa_layout = f.foa_layout, fob_layout = f.fob_layout;
  const uint8_t *foa_codes = f.foa_codes, *foa_sf = f.foa_sf, *fob_codes = f.fob_codes, *fob_sf = f.fob_sf;
  const float *foa_ts = f.foa_ts, *sa = f.sa, *fob_ts = f.fob_ts, *sb = f.sb, *__restrict__ pm = f.pm, *res_a_ts = f.res_a_ts, *res_b_ts = f.res_b_ts;
  float *__restrict__ lcat = f.lcat, *__restrict__ rcat = f.rcat;
  __nv_bfloat16 *__restrict__ lx = f.lx, *__restrict__ rx = f.rx;
  __shared__ float ps[32 * J][32 * J];
  __shared__ float fa[8][32 * J][R];                            // Fo_a sa of a warp's rows
  metis_pdl_wait();
  metis_pdl_trigger();                                      // the large GEMM behind this kernel sets itself up meanwhile
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int kc = ka + kb;
  const int64_t i0 = ((int64_t)((int)blockIdx.x - (is_first ? 0 : n_first)) * 8 + warp) * R;
  // An extent is a multiple of 64 where that side has factors (they are quantized in blocks along it); a plain operand may have any number of
  // rows, so each of the warp's rows is held against its extent.
  const int rows_m = (int)max(min(M - i0, (int64_t)R), (int64_t)0), rows_n = (int)max(min(N - i0, (int64_t)R), (int64_t)0);
  // ---- loads (ka, kb <= 64: two vectors per lane and operand) ----
  uint32_t a_code[J] = {}, a_sfb[J] = {}, b_code[J] = {}, b_sfb[J] = {};
  float sa_v[J] = {}, sb_v[J] = {}, g1[J][R] = {}, wt[J][R] = {};
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int u = lane + 32 * j;
    if (u < ka) {
      sa_v[j] = sa[u];
      if (rows_m > 0) {
        const uint8_t* src = foa_codes + (int64_t)u * (M / 2) + i0 / 2;
        a_code[j] = R == 4 ? src[0] | (uint32_t)src[1] << 8 : (R == 2 ? src[0] : src[0] >> (4 * (int)(i0 & 1)));
        a_sfb[j] = foa_sf[metis_sf_offset(u, i0 / 16, M / 16, foa_layout)];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) if (r < rows_n) wt[j][r] = rcat[(i0 + r) * kc + kb + u];
    }
    if (u < kb) {
      sb_v[j] = sb[u];
#pragma unroll
      for (int r = 0; r < R; ++r) if (r < rows_m) g1[j][r] = lcat[(i0 + r) * kc + u];
      if (rows_n > 0) {
        const uint8_t* src = fob_codes + (int64_t)u * (N / 2) + i0 / 2;
        b_code[j] = R == 4 ? src[0] | (uint32_t)src[1] << 8 : (R == 2 ? src[0] : src[0] >> (4 * (int)(i0 & 1)));
        b_sfb[j] = fob_sf[metis_sf_offset(u, i0 / 16, N / 16, fob_layout)];
      }
    }
  }
  const float tsa = ka ? *foa_ts : 0.0f, tsb = kb ? *fob_ts : 0.0f;
  const float inv_alpha = lx != nullptr ? 1.0f / ((*res_a_ts) * (*res_b_ts)) : 0.0f;
  for (int o = warp; o < ka; o += 32) {                     // four rows of P in flight
    float v[4][J];
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int j = 0; j < J; ++j) v[b][j] = o + 8 * b < ka && lane + 32 * j < kb ? pm[(o + 8 * b) * kb + lane + 32 * j] : 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int j = 0; j < J; ++j) if (o + 8 * b < ka) ps[o + 8 * b][lane + 32 * j] = v[b][j];
  }
  float raw_a[J][R], raw_b[J][R];                           // the factors as E2M1 x E4M3 products (exact in FP16), before any FP32 scale
  auto dequantize = [](uint32_t code, uint32_t sf, float (&out)[R]) {
    const __half2 sc = __float2half2_rn(metis_e4m3_value(sf));
#pragma unroll
    for (int r = 0; r < R; r += 2) {
      const float2 v = __half22float2(__hmul2(e2m1x2_to_half2(code >> (4 * r)), sc));
      out[r] = v.x;
      if (r + 1 < R) out[r + 1] = v.y;
    }
  };
#pragma unroll
  for (int j = 0; j < J; ++j) {
    dequantize(a_code[j], a_sfb[j], raw_a[j]);
    dequantize(b_code[j], b_sfb[j], raw_b[j]);
#pragma unroll
    for (int r = 0; r < R; ++r) fa[warp][lane + 32 * j][r] = raw_a[j][r] * tsa * sa_v[j];
  }
  __syncthreads();
  if (rows_m > 0) {
#pragma unroll 4
    for (int u = 0; u < ka; ++u) {
      float fr[R];
#pragma unroll
      for (int r = 0; r < R; ++r) fr[r] = fa[warp][u][r];
#pragma unroll
      for (int j = 0; j < J; ++j)
        {
          const float p = ps[u][lane + 32 * j];
#pragma unroll
          for (int r = 0; r < R; ++r) g1[j][r] = fmaf(fr[r], p, g1[j][r]);
        }
    }
  }
  const float l_scale = tsb * inv_alpha, r_scale = tsa * inv_alpha;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t i = i0 + r;
    const bool in_m = r < rows_m, in_n = r < rows_n;
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const int u = lane + 32 * j;
      const float a = g1[j][r] * sb_v[j];
      if (lx == nullptr) {
        if (in_m && u < kb) lcat[i * kc + u] = a;
        if (in_m && u < ka) lcat[i * kc + kb + u] = raw_a[j][r] * tsa * sa_v[j];
        if (in_n && u < kb) rcat[i * kc + u] = raw_b[j][r] * tsb;
        continue;
      }
      if (u < kb) {
        if (in_m) {
          const float v = a * l_scale;
          const __nv_bfloat16 h = __float2bfloat16_rn(v);
          lx[i * kx + u] = h;
          lx[i * kx + kb + u] = __float2bfloat16_rn(v - __bfloat162float(h));
        }
        if (in_n) rx[i * kx + u] = rx[i * kx + kb + u] = __float2bfloat16_rn(raw_b[j][r]);
      }
      if (u < ka) {
        if (in_m) lx[i * kx + 2 * kb + u] = lx[i * kx + 2 * kb + ka + u] = __float2bfloat16_rn(raw_a[j][r]);
        if (in_n) {
          const float v = wt[j][r] * sa_v[j] * r_scale;
          const __nv_bfloat16 h = __float2bfloat16_rn(v);
          rx[i * kx + 2 * kb + u] = h;
          rx[i * kx + 2 * kb + ka + u] = __float2bfloat16_rn(v - __bfloat162float(h));
        }
      }
    }
    for (int c = 2 * kc + lane; c < kx && lx != nullptr; c += 32) {
      if (in_m) lx[i * kx + c] = __float2bfloat16_rn(0.0f);
      if (in_n) rx[i * kx + c] = __float2bfloat16_rn(0.0f);
    }
  }
}

// Ranks above 64: the same finishing step as three kernels that tile over the rank.
//   lowrank_deq_wide_kernel    Lcat[:, kb:] = Fo_a sa and Rcat[:, :kb] = Fo_b from the NVFP4 factors (a thread
//                              dequantizes eight consecutive rows of one vector from one 32-bit load)
//   lowrank_gemm_wide_kernel   Lcat[:, :kb] = (G1 + Lcat[:, kb:] P) sb, a 64 x 64 x 16 tiled FP32 product, 4 x 4 per thread
//   lowrank_bf16_kernel        the BF16 correction operands, eight columns per thread
constexpr int LW_MAXK = 256;
__global__ void __launch_bounds__(256)
lowrank_deq_wide_kernel(const __grid_constant__ FinishArgs first, const __grid_constant__ FinishArgs second) {
  metis_pdl_wait();
  const FinishArgs& f = blockIdx.y == 0 ? first : second;
  const int64_t M = f.M, N = f.N;
  const int ka = f.ka, kb = f.kb, kx = f.kx, foa_layout = f.foa_layout, fob_layout = f.fob_layout;
  const uint8_t *foa_codes = f.foa_codes, *foa_sf = f.foa_sf, *fob_codes = f.fob_codes, *fob_sf = f.fob_sf;
  const float *foa_ts = f.foa_ts, *sa = f.sa, *fob_ts = f.fob_ts;
  float *__restrict__ lcat = f.lcat, *__restrict__ rcat = f.rcat;
  __nv_bfloat16 *__restrict__ lx = f.lx, *__restrict__ rx = f.rx;
  const int tid = threadIdx.x, kc = ka + kb;
  const int64_t i0 = (int64_t)blockIdx.x * 32 + 8 * (tid & 3);      // this thread's eight rows (an extent with factors is a multiple of 64)
  const float tsa = ka ? *foa_ts : 0.0f, tsb = kb ? *fob_ts : 0.0f;
  for (int u = tid >> 2; u < ka; u += 64) {
    if (i0 >= M) break;
    const uint32_t word = *reinterpret_cast<const uint32_t*>(foa_codes + (int64_t)u * (M / 2) + i0 / 2);
    const float sc = metis_e4m3_value(foa_sf[metis_sf_offset(u, i0 / 16, M / 16, foa_layout)]), su = sa[u];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float raw = metis_e2m1_value((word >> (4 * j)) & 15u) * sc;
      lcat[(i0 + j) * kc + kb + u] = raw * tsa * su;
      if (lx != nullptr) {                                  // the exact factor entry, both of its column groups
        const __nv_bfloat16 e = __float2bfloat16_rn(raw);
        lx[(i0 + j) * kx + 2 * kb + u] = e;
        lx[(i0 + j) * kx + 2 * kb + ka + u] = e;
      }
    }
  }
  for (int t = tid >> 2; t < kb; t += 64) {
    if (i0 >= N) break;
    const uint32_t word = *reinterpret_cast<const uint32_t*>(fob_codes + (int64_t)t * (N / 2) + i0 / 2);
    const float sc = metis_e4m3_value(fob_sf[metis_sf_offset(t, i0 / 16, N / 16, fob_layout)]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float raw = metis_e2m1_value((word >> (4 * j)) & 15u) * sc;
      rcat[(i0 + j) * kc + t] = raw * tsb;
      if (rx != nullptr) {
        const __nv_bfloat16 e = __float2bfloat16_rn(raw);
        rx[(i0 + j) * kx + t] = e;
        rx[(i0 + j) * kx + kb + t] = e;
      }
    }
  }
}

__global__ void __launch_bounds__(256)
lowrank_gemm_wide_kernel(const __grid_constant__ FinishArgs first, const __grid_constant__ FinishArgs second) {
  metis_pdl_wait();
  const FinishArgs& f = blockIdx.z == 0 ? first : second;
  const int64_t M = f.M;
  const int ka = f.ka, kb = f.kb;
  const float *__restrict__ sb = f.sb, *__restrict__ pm = f.pm;
  float* __restrict__ lcat = f.lcat;
  if ((int)blockIdx.x * 64 >= kb || (int64_t)blockIdx.y * 64 >= M) return;
  constexpr int KT = 16;
  __shared__ __align__(16) float as[KT][68], bs[KT][68];   // [u][row], [u][column]
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, kc = ka + kb;
  const int64_t m0 = (int64_t)blockIdx.y * 64;
  const int n0 = blockIdx.x * 64;
  float acc[4][4] = {};
  for (int u0 = 0; u0 < ka; u0 += KT) {
    __syncthreads();
    for (int o = tid; o < 64 * KT; o += 256) {
      const int uu = o % KT, r = o / KT;                    // consecutive threads: consecutive u of one row (contiguous in Lcat)
      as[uu][r] = (m0 + r < M && u0 + uu < ka) ? lcat[(m0 + r) * kc + kb + u0 + uu] : 0.0f;
      const int t = o % 64, u2 = o / 64;                    // consecutive threads: consecutive columns of one row of P
      bs[u2][t] = (u0 + u2 < ka && n0 + t < kb) ? pm[(int64_t)(u0 + u2) * kb + n0 + t] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int uu = 0; uu < KT; ++uu) {
      const float4 a = *reinterpret_cast<const float4*>(&as[uu][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&bs[uu][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t r = m0 + ty * 4 + i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int t = n0 + tx * 4 + j;
      if (t < kb) lcat[r * kc + t] = (lcat[r * kc + t] + acc[i][j]) * sb[t];
    }
  }
}

// Then the general halves of the BF16 correction operands (the layout of lowrank_finish_kernel): [A hi | A lo] of Lx and
// [B hi | B lo] of Rx from the finished FP32 operands, and the zero padding up to kx columns; the exact factor groups
// were written by lowrank_deq_wide_kernel.  One thread per row and eight columns (the group boundaries 2 k_b and
// 2 (k_a + k_b) are multiples of eight).
__global__ void __launch_bounds__(256)
lowrank_bf16_kernel(const __grid_constant__ FinishArgs first, const __grid_constant__ FinishArgs second) {
  metis_pdl_wait();
  const FinishArgs& f = blockIdx.y == 0 ? first : second;
  const int64_t M = f.M, N = f.N;
  const int ka = f.ka, kb = f.kb, kx = f.kx;
  const float *__restrict__ lcat = f.lcat, *__restrict__ rcat = f.rcat, *foa_ts = f.foa_ts, *__restrict__ sa = f.sa, *fob_ts = f.fob_ts, *res_a_ts = f.res_a_ts, *res_b_ts = f.res_b_ts;
  __nv_bfloat16 *__restrict__ lx = f.lx, *__restrict__ rx = f.rx;
  if (lx == nullptr) return;                                // a layer of fewer than 256 rows beside one that has them
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t mx = M > N ? M : N;
  const int per_row = kx / 8, kc = ka + kb;
  if (idx >= mx * per_row) return;
  const int64_t i = idx / per_row;
  const int c0 = (int)(idx - i * per_row) * 8;
  const float inv_alpha = 1.0f / ((*res_a_ts) * (*res_b_ts));
  const float l_scale = (kb ? *fob_ts : 0.0f) * inv_alpha, r_scale = (ka ? *foa_ts : 0.0f) * inv_alpha;
  __align__(16) __nv_bfloat16 o[8];
  if (c0 < 2 * kb) {                                        // [A hi | A lo]
    if (i < M) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c0 + e, t = c < kb ? c : c - kb;
        const float v = lcat[i * kc + t] * l_scale;
        const float h = __bfloat162float(__float2bfloat16_rn(v));
        o[e] = __float2bfloat16_rn(c < kb ? h : v - h);
      }
      *reinterpret_cast<uint4*>(lx + i * kx + c0) = *reinterpret_cast<const uint4*>(o);
    }
  } else if (c0 < 2 * kc) {                                 // [B hi | B lo]
    if (i < N) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int u0 = c0 + e - 2 * kb, u = u0 < ka ? u0 : u0 - ka;
        const float v = rcat[i * kc + kb + u] * sa[u] * r_scale;
        const float h = __bfloat162float(__float2bfloat16_rn(v));
        o[e] = __float2bfloat16_rn(u0 < ka ? h : v - h);
      }
      *reinterpret_cast<uint4*>(rx + i * kx + c0) = *reinterpret_cast<const uint4*>(o);
    }
  } else {                                                  // padding of both operands
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    if (i < M) *reinterpret_cast<uint4*>(lx + i * kx + c0) = z;
    if (i < N) *reinterpret_cast<uint4*>(rx + i * kx + c0) = z;
  }
}

// out = y0 + Lcat Rcat^T, 64 x 64 tile per CTA
__global__ void __launch_bounds__(256)
rank_update_kernel(const float* __restrict__ y0, int64_t M, int64_t N, int kc, const float* __restrict__ lcat,
                   const float* __restrict__ rcat, void* __restrict__ out, int out_dtype, int64_t ldo) {
  metis_pdl_wait();
  extern __shared__ __align__(16) float sm[];
  float* ls = sm;                       // [kc][64 + 4]
  float* rs = sm + kc * 68;
  const int tid = threadIdx.x;
  const int64_t m0 = (int64_t)blockIdx.y * 64, n0 = (int64_t)blockIdx.x * 64;
  for (int i = tid; i < 64 * kc; i += 256) {
    const int r = i / kc, t = i % kc;
    ls[t * 68 + r] = (m0 + r < M) ? lcat[(m0 + r) * kc + t] : 0.0f;
    rs[t * 68 + r] = (n0 + r < N) ? rcat[(n0 + r) * kc + t] : 0.0f;
  }
  __syncthreads();
  const int ty = tid >> 4, tx = tid & 15;
  float acc[4][4] = {};
  for (int t = 0; t < kc; ++t) {
    const float4 a = *reinterpret_cast<const float4*>(ls + t * 68 + ty * 4);
    const float4 b = *reinterpret_cast<const float4*>(rs + t * 68 + tx * 4);
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t r = m0 + ty * 4 + i, c = n0 + tx * 4 + j;
      if (r < M && c < N) {
        const float v = y0[r * N + c] + acc[i][j];
        if (out_dtype == METIS_BF16) reinterpret_cast<__nv_bfloat16*>(out)[r * ldo + c] = __float2bfloat16_rn(v);
        else reinterpret_cast<float*>(out)[r * ldo + c] = v;
      }
    }
}


// ------------------------------------------------------------------------------------------------
// Gradients of the weight factors (Section 3.2, the derivatives listed after Eq. 3).  With the weight gradient
// G (n x m, FP32 or BF16, as produced by the wgrad product) and a dequantized factor F stored k x len:
//   TRANS = 0:  out[t][r] = scale_t * sum_c G[r][c] F[t][c]      (r over n, c over m:  dL/dV from U)
//   TRANS = 1:  out[t][r] = scale_t * sum_c G[c][r] F[t][c]      (r over m, c over n:  dL/dU from V)
// scale_t = sigma_t.  With `other` given (the factor lying along r), a strip also writes its partial of
//   dsigma[t] = sum_r other[t][r] * (sum_c ...)   to ds_part[strip][t].
//
// A contraction whose large operand is read once: bound by the bytes of G.  A factor entry without its tensor scale
// is an E2M1 x E4M3 product and exact in BF16, an FP32 gradient is three BF16 terms, so the products of mma.sync are
// exact and only the FP32 sums round.  The tensor core truncates its sums, so an accumulator runs over a quarter of a chunk (6 adds)
// and is then added to an FP32 total.  A CTA owns a strip of 64 values of r; its eight warps are 2 (r) x 4 (quarters of a
// chunk of 128 values of c), and the CTAs of a cluster divide the chunks; the 4 * cluster totals of a strip are added in a
// fixed order at the end (shared memory, then distributed shared memory).
// G comes through a ring of asynchronous copies (three FP32 chunks, five BF16 ones, in flight: 96 and 80 KB per SM; loads straight into
// fragment registers, two steps ahead of twelve warps, left every warp waiting for memory four cycles in seven), the factor
// chunk through registers a chunk ahead and, dequantized, through a double buffer; the contraction index (and, for TRANS, r) is permuted so that
// a fragment load is four neighbours.  14336 x 4096 FP32, k = 32: 140 -> 102 us (TRANS = 0), 154 -> 76 us; a chunk of 32 KB takes
// 1.45 us of an SM with two warps per scheduler, twice what its bytes take.
constexpr int FG_ROWS = 64, FG_CHUNK = 128, FG_KW = FG_CHUNK / 32, FG_THREADS = 64 * FG_KW, FG_PITCH = FG_CHUNK + 16;    // pitch: 8 words mod 32, conflict-free 64-bit fragment loads
constexpr int FG_QUADS = FG_ROWS * FG_CHUNK / 4 / FG_THREADS;                    // groups of four elements per thread and chunk
__host__ __device__ constexpr int fg_stages(int es) { return es == 4 ? 4 : 6; }                      // chunks of G in flight or in use: 128 KB (FP32), 96 KB
// Dynamic shared memory of a CTA that works on `per` chunks: the factor's double buffer and the ring, or the sums at the end, which take their place.
// A ring no longer than its chunks lets two CTAs share an SM, so that clusters of eight find room at once (1024 x 1024, k = 8, with the
// whole ring: 14.2 + 11.9 us for the two gradients, 8.7 + 7.7 so, 8.9 + 8.4 with loads straight into registers).
constexpr int fg_smem(int nt, int es, int per) {
  const int ring = 2 * 8 * nt * FG_PITCH * 2 + (per < fg_stages(es) ? per : fg_stages(es)) * FG_ROWS * FG_CHUNK * es, red = FG_KW * FG_ROWS * (8 * nt + 1) * 4;
  return ring > red ? ring : red;
}

__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// the next BF16 term of a pair of floats; x and y become what is left
__device__ __forceinline__ uint32_t take_bf16x2(float& x, float& y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  const uint32_t w = *reinterpret_cast<const uint32_t*>(&h);
  x -= __uint_as_float(w << 16);
  y -= __uint_as_float(w & 0xFFFF0000u);
  return w;
}
// four consecutive elements of G into shared memory, zeros unless `in` (src is a valid address all the same; VEC: 16-byte aligned FP32, 8-byte aligned BF16, asynchronous)
template <typename T, bool VEC>
__device__ __forceinline__ void fg_fetch4(uint32_t dst, const T* src, bool in) {
  if (VEC) {
    if (sizeof(T) == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(in ? 16 : 0) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(in ? 8 : 0) : "memory");
  } else {
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (in) {
#pragma unroll
      for (int e = 0; e < 4; ++e) w[e] = sizeof(T) == 4 ? reinterpret_cast<const uint32_t*>(src)[e] : (uint32_t)reinterpret_cast<const uint16_t*>(src)[e];
    }
    if (sizeof(T) == 4) asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]) : "memory");
    else asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(dst), "r"(w[0] | (w[1] << 16)), "r"(w[2] | (w[3] << 16)) : "memory");
  }
}


// One entry of the contraction as FP32 multiply-adds in order.  An FP32 gradient that is infinite or rounds to infinity in BF16
// leaves a NaN as its remainder, and sums that overflow may meet with opposite signs: an entry that came out as a NaN is
// settled here, so that the gradients are infinite where FP32 products make them so and a NaN stands for a real one.  Never
// entered for finite gradients; a NaN ends the sum.
template <typename T>
__device__ __noinline__ float fg_plain_sum(const T* g, int64_t stride, int64_t n_c, const uint8_t* f_codes, const uint8_t* f_sf, int f_layout, int64_t t) {
  float acc = 0.0f;
  for (int64_t c = 0; c < n_c && !isnan(acc); ++c) acc = fmaf((float)g[c * stride], deq_at(f_codes, f_sf, f_layout, n_c, t, c), acc);
  return acc;
}

template <int NT, bool TRANS, typename T, bool VEC>     // NT = ceil(k / 8) groups of eight factor vectors, at most 8
__global__ void __launch_bounds__(FG_THREADS, 1)
factor_grad_kernel(const T* __restrict__ gsrc, int64_t ldg, int64_t n_r, int64_t n_c, int k, int t0, int k_all,
                   const uint8_t* f_codes, const uint8_t* f_sf, int f_layout, const float* f_ts,
                   const uint8_t* o_codes, const uint8_t* o_sf, int o_layout, const float* o_ts,
                   const float* __restrict__ sigma, float* __restrict__ out, float* __restrict__ ds_part) {
  // factor vectors t0 .. t0 + k - 1 of k_all (a launch handles at most 64 of them)
  extern __shared__ __align__(16) unsigned char fg_sm[];
  constexpr int QB = 4 * (int)sizeof(T), STAGES = fg_stages(sizeof(T)), STAGE = FG_ROWS * FG_CHUNK * (int)sizeof(T);
  __nv_bfloat16* fs = reinterpret_cast<__nv_bfloat16*>(fg_sm);                   // [2][8 NT][FG_PITCH]
  unsigned char* ring = fg_sm + 2 * 8 * NT * FG_PITCH * 2;                       // [STAGES, or fewer chunks][FG_ROWS x FG_CHUNK of G]
  float* red = reinterpret_cast<float*>(fg_sm);                                  // [FG_KW][FG_ROWS][8 NT + 1], after the loop
  constexpr int RP = 8 * NT + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
  const int mw = warp & 1, kw = warp >> 1;
  uint32_t rank, csize;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(csize));
  const int64_t strip = blockIdx.x / csize;
  const int chunks = (int)((n_c + FG_CHUNK - 1) / FG_CHUNK), per = (chunks + (int)csize - 1) / (int)csize;
  const int ch0 = (int)rank * per, ch1 = min(chunks, ch0 + per);
  const int64_t c_stride = TRANS ? ldg : 1;

  // A chunk lies in the ring as it lies in memory: FG_ROWS rows of 32 quads of c, or (TRANS) FG_CHUNK rows of 16 quads of r.  Quad i of
  // row j is stored at i ^ 4 (j & 3), or i ^ SW ((j >> 2) & 3): the 128 bytes that a fragment load of eight (FP32) or sixteen lanes
  // collects from two or four rows then lie in different banks.
  constexpr int SW = sizeof(T) == 4 ? 2 : 4;
  // This thread's quads: column i of rows j0, j0 + FJ, ...  (FJ is a multiple of what the swizzle looks at.)
  constexpr int FJ = TRANS ? FG_THREADS / 16 : FG_THREADS / 32;
  const int fj = TRANS ? tid >> 4 : tid >> 5, fi = TRANS ? tid & 15 : tid & 31;
  const uint32_t f_dst = (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)(TRANS ? fj * 16 + (fi ^ (SW * ((fj >> 2) & 3))) : fj * 32 + (fi ^ (4 * (fj & 3)))) * QB;
  const int64_t f_r = strip * FG_ROWS + (TRANS ? 4 * fi : fj);                   // first r of the first quad
  const int f_rows = (int)min((int64_t)FG_ROWS, n_r - f_r), f_c = TRANS ? fj : 4 * fi;
  auto fetch = [&](int ch) {
    const uint32_t dst = f_dst + (uint32_t)((ch - ch0) % STAGES) * STAGE;
    const int64_t c0 = (int64_t)ch * FG_CHUNK + f_c;
    const T* src = gsrc + f_r * (TRANS ? 1 : ldg) + c0 * c_stride;
    const int c_left = (int)min((int64_t)FG_CHUNK, n_c - c0);
#pragma unroll
    for (int u = 0; u < FG_QUADS; ++u) {
      const bool in = TRANS ? f_rows > 0 && FJ * u < c_left : FJ * u < f_rows && c_left > 0;
      fg_fetch4<T, VEC>(dst + u * FJ * (TRANS ? 16 : 32) * QB, in ? src + (int64_t)(FJ * u) * ldg : gsrc, in);
    }
  };
  // A step is 16 values of c: slots {2q, 2q+1, 2q+8, 2q+9} of a fragment hold c = base + 4q .. 4q + 3.
  //   TRANS = 0: one load is four values of c of row 32 mw + 16 i + g (+ 8)
  //   TRANS = 1: one load is rows 32 mw + 4g .. 4g + 3 of one c; rows g / g + 8 of fragment i are 4g + 2i / + 1
  auto load_step = [&](const unsigned char* st, float4 (&v)[4], int c0) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = TRANS ? c0 + 4 * q + u : 32 * mw + 16 * (u >> 1) + 8 * (u & 1) + g;
      const int at = TRANS ? j * 16 + ((8 * mw + g) ^ (SW * q)) : j * 32 + (((c0 >> 2) + q) ^ (4 * (j & 3)));
      if (sizeof(T) == 4) v[u] = *reinterpret_cast<const float4*>(st + at * QB);
      else {
        const uint2 w = *reinterpret_cast<const uint2*>(st + at * QB);
        v[u] = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xFFFF0000u));
      }
    }
  };
  const bool wide_codes = (reinterpret_cast<uintptr_t>(f_codes) & 7u) == 0;      // n_c is a multiple of 16: every block is then aligned
  // Factor chunk: codes and scales travel in registers for a chunk (8 NT x 8 blocks, one or two per thread) and are dequantized without the
  // tensor scale on the way into shared memory; rows beyond k and values of c beyond n_c are zero.
  constexpr int FB = (8 * NT * (FG_CHUNK / 16) + FG_THREADS - 1) / FG_THREADS;
  uint2 code[FB];
  uint32_t scale[FB];
  auto fetch_factor = [&](int ch) {
#pragma unroll
    for (int u = 0; u < FB; ++u) {
      const int o = tid + FG_THREADS * u, t = o / (FG_CHUNK / 16);
      const int64_t c = (int64_t)ch * FG_CHUNK + 16 * (o % (FG_CHUNK / 16));
      code[u] = make_uint2(0u, 0u); scale[u] = 0u;
      if (t < k && c < n_c) {
        const uint8_t* src = f_codes + (int64_t)(t0 + t) * (n_c / 2) + c / 2;
        if (wide_codes) code[u] = *reinterpret_cast<const uint2*>(src);
        else code[u] = make_uint2(src[0] | (src[1] << 8) | (src[2] << 16) | ((uint32_t)src[3] << 24), src[4] | (src[5] << 8) | (src[6] << 16) | ((uint32_t)src[7] << 24));
        scale[u] = f_sf[metis_sf_offset(t0 + t, c / 16, n_c / 16, f_layout)];
      }
    }
  };
  auto store_factor = [&](int buf) {
#pragma unroll
    for (int u = 0; u < FB; ++u) {
      const int o = tid + FG_THREADS * u, t = o / (FG_CHUNK / 16), b = o % (FG_CHUNK / 16);
      if (8 * NT * (FG_CHUNK / 16) % FG_THREADS != 0 && t >= 8 * NT) continue;
      uint32_t w[8];
      // E2M1 pairs to FP16 in one conversion; the products with the block scale have six significant bits and lie
      // between 2^-10 and 2688, so they are exact in FP16 and in BF16
      const __half2 sc = __float2half2_rn(metis_e4m3_value(scale[u]));
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float2 v = __half22float2(__hmul2(e2m1x2_to_half2((j < 4 ? code[u].x : code[u].y) >> (8 * (j & 3))), sc));
        const __nv_bfloat162 h = __floats2bfloat162_rn(v.x, v.y);
        w[j] = *reinterpret_cast<const uint32_t*>(&h);
      }
      uint4* dst = reinterpret_cast<uint4*>(fs + (buf * 8 * NT + t) * FG_PITCH + 16 * b);
      dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
      dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
  };
  float acc[2][NT][4], total[2][NT][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = total[i][j][e] = 0.0f;
#pragma unroll
  for (int p = 0; p < STAGES - 1; ++p) {
    if (ch0 + p < ch1) fetch(ch0 + p);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  if (ch0 < ch1) {
    fetch_factor(ch0);
    store_factor(0);
    if (ch0 + 1 < ch1) fetch_factor(ch0 + 1);
  }
  for (int ch = ch0; ch < ch1; ++ch) {
    const int buf = (ch - ch0) & 1;
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();                                       // chunk ch is there; what held chunk ch - 1 may be overwritten
    if (ch + STAGES - 1 < ch1) fetch(ch + STAGES - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (ch + 1 < ch1) store_factor(buf ^ 1);
    if (ch + 2 < ch1) fetch_factor(ch + 2);
    const unsigned char* st_g = ring + ((ch - ch0) % STAGES) * STAGE;
    float4 vv[2][4];
    load_step(st_g, vv[0], 32 * kw);
    load_step(st_g, vv[1], 32 * kw + 16);
#pragma unroll
    for (int st = 0; st < 2; ++st) {
      const int c_w = 32 * kw + 16 * st;
      const float4 (&v)[4] = vv[st];
      float ax[2][4][2];                                                         // [fragment][register][pair]
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (TRANS) {
          const float* e0 = reinterpret_cast<const float*>(&v[0]) + 2 * i; const float* e1 = reinterpret_cast<const float*>(&v[1]) + 2 * i;
          const float* e2 = reinterpret_cast<const float*>(&v[2]) + 2 * i; const float* e3 = reinterpret_cast<const float*>(&v[3]) + 2 * i;
          ax[i][0][0] = e0[0]; ax[i][0][1] = e1[0]; ax[i][1][0] = e0[1]; ax[i][1][1] = e1[1];
          ax[i][2][0] = e2[0]; ax[i][2][1] = e3[0]; ax[i][3][0] = e2[1]; ax[i][3][1] = e3[1];
        } else {
          ax[i][0][0] = v[2 * i].x; ax[i][0][1] = v[2 * i].y; ax[i][1][0] = v[2 * i + 1].x; ax[i][1][1] = v[2 * i + 1].y;
          ax[i][2][0] = v[2 * i].z; ax[i][2][1] = v[2 * i].w; ax[i][3][0] = v[2 * i + 1].z; ax[i][3][1] = v[2 * i + 1].w;
        }
      }
      uint32_t bf[NT][2];
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const uint2 w = *reinterpret_cast<const uint2*>(fs + (buf * 8 * NT + 8 * j + g) * FG_PITCH + c_w + 4 * q);
        bf[j][0] = w.x; bf[j][1] = w.y;
      }
#pragma unroll
      for (int term = 0; term < (sizeof(T) == 4 ? 3 : 1); ++term) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          uint32_t a[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) a[e] = take_bf16x2(ax[i][e][0], ax[i][e][1]);
#pragma unroll
          for (int j = 0; j < NT; ++j) mma_16816(acc[i][j], a, bf[j][0], bf[j][1]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) { total[i][j][e] += acc[i][j][e]; acc[i][j][e] = 0.0f; }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();                                         // the ring has been read
  // ---- sums of the quarters of a chunk, then of the cluster's CTAs ----
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int row = 32 * mw + (TRANS ? 4 * g + 2 * i + (e >> 1) : 16 * i + g + 8 * (e >> 1));
        red[(kw * FG_ROWS + row) * RP + 8 * j + 2 * q + (e & 1)] = total[i][j][e];
      }
  __syncthreads();
  for (int o = tid; o < FG_ROWS * 8 * NT; o += FG_THREADS) {
    const int row = o / (8 * NT), t = o % (8 * NT);
    float v = red[row * RP + t];
#pragma unroll
    for (int w = 1; w < FG_KW; ++w) v += red[(w * FG_ROWS + row) * RP + t];
    red[row * RP + t] = v;
  }
  asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
  // CTA `rank` finishes the factor vectors t = rank, rank + csize, ..., one warp per vector
  const float fts = *f_ts, ots = ds_part != nullptr ? *o_ts : 0.0f;
  const uint32_t red_addr = (uint32_t)__cvta_generic_to_shared(red);
  for (int t = (int)rank + (int)csize * warp; t < k; t += (int)csize * (FG_THREADS / 32)) {
    float ds = 0.0f;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = lane + 32 * h;
      const int64_t r = strip * FG_ROWS + row;
      float v = 0.0f;
      for (uint32_t c = 0; c < csize; ++c) {
        uint32_t peer;
        float x;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(red_addr + (uint32_t)(row * RP + t) * 4u), "r"(c));
        asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(x) : "r"(peer));
        v += x;
      }
      if (isnan(v) && r < n_r) v = fg_plain_sum<T>(gsrc + (TRANS ? r : r * ldg), c_stride, n_c, f_codes, f_sf, f_layout, t0 + t);
      v *= fts;
      if (r < n_r) {
        out[(int64_t)(t0 + t) * n_r + r] = v * sigma[t0 + t];
        if (ds_part != nullptr) ds += v * deq_at(o_codes, o_sf, o_layout, n_r, t0 + t, r) * ots;
      }
    }
    if (ds_part != nullptr) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ds += __shfl_xor_sync(0xFFFFFFFFu, ds, o);
      if (lane == 0) ds_part[strip * k_all + t0 + t] = ds;
    }
  }
  asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");   // peers may still be reading
}

// dsigma[t] = sum over the partials, one warp per t (each lane every 32nd partial, then a fixed tree)
__global__ void __launch_bounds__(256)
factor_grad_sigma_kernel(const float* __restrict__ part, int n_part, int k, float* __restrict__ ds) {
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= k) return;
  float v = 0.0f;
  for (int i = lane; i < n_part; i += 32) v += part[(int64_t)i * k + t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  if (lane == 0) ds[t] = v;
}

template <int NT, bool TRANS, typename T, bool VEC>
metis_status_t launch_factor_grad_nt(cudaStream_t s, const T* g, int64_t ldg, int64_t n_r, int64_t n_c, int kg, int t0, int k, const metis_nvfp4_t* f,
                                     const metis_nvfp4_t* o, const float* sigma, float* out, float* ds_part) {
  // CTAs of a cluster divide the contraction until three quarters of the SMs have one (a strip's work is the whole contraction; an SM
  // alone fetches about twice its share of the memory's bandwidth, so that a partly filled wave costs little)
  const int64_t strips = metis_ceil_div(n_r, FG_ROWS), chunks = metis_ceil_div(n_c, FG_CHUNK);
  unsigned csize = 1;
  while (csize < 8 && strips * csize < 111 && 2 * csize <= chunks) csize *= 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(strips * csize)); cfg.blockDim = dim3(FG_THREADS); cfg.stream = s;
  cfg.dynamicSmemBytes = (size_t)fg_smem(NT, sizeof(T), (int)metis_ceil_div(chunks, (int64_t)csize));
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = csize; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  METIS_CUDA_TRY(cudaLaunchKernelEx(&cfg, factor_grad_kernel<NT, TRANS, T, VEC>, g, ldg, n_r, n_c, kg, t0, k, (const uint8_t*)f->codes, (const uint8_t*)f->scales,
      (int)f->sf_layout, (const float*)f->tensor_scale, (const uint8_t*)(o ? o->codes : nullptr), (const uint8_t*)(o ? o->scales : nullptr),
      (int)(o ? o->sf_layout : 0), (const float*)(o ? o->tensor_scale : nullptr), sigma, out, ds_part));
  METIS_COUNT_LAUNCH();
  return METIS_OK;
}

template <bool TRANS, typename T, bool VEC>
metis_status_t launch_factor_grad_t(cudaStream_t s, const T* g, int64_t ldg, int64_t n_r, int64_t n_c, int k, const metis_nvfp4_t* f, const metis_nvfp4_t* o,
                                    const float* sigma, float* out, float* ds_part) {
  for (int t0 = 0; t0 < k; t0 += 64) {                  // at most 64 factor vectors per pass over the gradient
    const int kg = k - t0 < 64 ? k - t0 : 64;
#define METIS_FG(NT) METIS_TRY((launch_factor_grad_nt<NT, TRANS, T, VEC>(s, g, ldg, n_r, n_c, kg, t0, k, f, o, sigma, out, ds_part)))
    if (kg <= 8) METIS_FG(1);
    else if (kg <= 16) METIS_FG(2);
    else if (kg <= 32) METIS_FG(4);
    else if (kg <= 48) METIS_FG(6);
    else METIS_FG(8);
#undef METIS_FG
  }
  return METIS_OK;
}

template <bool TRANS>
metis_status_t launch_factor_grad(cudaStream_t s, const void* g, int g_dtype, int64_t ldg, int64_t n_r, int64_t n_c, int k,
                                  const metis_nvfp4_t* f, const metis_nvfp4_t* o, const float* sigma, float* out, float* ds_part) {
  // four elements per load when every row starts on the boundary of such a load; element by element otherwise
  if (g_dtype == METIS_BF16) {
    const __nv_bfloat16* gb = reinterpret_cast<const __nv_bfloat16*>(g);
    const bool vec = (reinterpret_cast<uintptr_t>(g) & 7u) == 0 && ldg % 4 == 0;
    return vec ? launch_factor_grad_t<TRANS, __nv_bfloat16, true>(s, gb, ldg, n_r, n_c, k, f, o, sigma, out, ds_part)
               : launch_factor_grad_t<TRANS, __nv_bfloat16, false>(s, gb, ldg, n_r, n_c, k, f, o, sigma, out, ds_part);
  }
  const float* gf = reinterpret_cast<const float*>(g);
  const bool vec = metis_aligned16(g) && ldg % 4 == 0;
  return vec ? launch_factor_grad_t<TRANS, float, true>(s, gf, ldg, n_r, n_c, k, f, o, sigma, out, ds_part)
             : launch_factor_grad_t<TRANS, float, false>(s, gf, ldg, n_r, n_c, k, f, o, sigma, out, ds_part);
}

// the host-side checks of factor_grads, callable before anything is enqueued
metis_status_t factor_grads_check(const metis_operand_t* w, const float* d_left, const float* d_sigma, const void* ws, size_t ws_bytes) {
  if (!w || w->k <= 0 || w->k > LW_MAXK || !w->sigma) return METIS_ERR_SHAPE;
  const metis_nvfp4_t *lq = &w->left_q, *rq = &w->right_q;
  if (!lq->codes || !rq->codes || lq->k_len != w->rows || rq->k_len != w->cols) return METIS_ERR_SHAPE;
  if (d_sigma && !d_left) return METIS_ERR_INVALID_ARG;          // the sigma partials ride on the d_left pass
  if (d_sigma && (!ws || ws_bytes < sizeof(float) * (size_t)metis_ceil_div(w->rows, FG_ROWS) * w->k)) return METIS_ERR_WORKSPACE;
  return METIS_OK;
}

// d_left (k x n), d_sigma (k), d_right (k x m) of the weight operand W_t = left diag(sigma) right^T from dw (n x m).
metis_status_t factor_grads(metis_context* ctx, const void* dw, int dw_dtype, int64_t lddw, const metis_operand_t* w,
                            float* d_left, float* d_sigma, float* d_right, void* ws, size_t ws_bytes, cudaStream_t s) {
  (void)ctx;
  if (!w || w->k <= 0 || w->k > LW_MAXK || !w->sigma) return METIS_ERR_SHAPE;
  const int64_t n = w->rows, m = w->cols;
  const metis_nvfp4_t *lq = &w->left_q, *rq = &w->right_q;
  if (!lq->codes || !rq->codes || lq->k_len != n || rq->k_len != m) return METIS_ERR_SHAPE;
  const int64_t n_part = metis_ceil_div(n, FG_ROWS);
  if (d_sigma && (!ws || ws_bytes < sizeof(float) * (size_t)n_part * w->k)) return METIS_ERR_WORKSPACE;
  float* part = reinterpret_cast<float*>(ws);
  // dL/dV (the paper's V = left, n x k): rows of dw against U = right; also the partials of dL/dS
  if (d_left || d_sigma) {
    if (!d_left) return METIS_ERR_INVALID_ARG;          // the sigma partials ride on the d_left pass
    METIS_TRY(launch_factor_grad<false>(s, dw, dw_dtype, lddw, n, m, w->k, rq, d_sigma ? lq : nullptr, w->sigma, d_left,
                                        d_sigma ? part : nullptr));
    if (d_sigma) {
      factor_grad_sigma_kernel<<<(unsigned)metis_ceil_div(w->k, 8), 256, 0, s>>>(part, (int)n_part, w->k, d_sigma); METIS_COUNT_LAUNCH();
      METIS_CUDA_TRY(cudaGetLastError());
    }
  }
  // dL/dU (the paper's U = right, m x k): columns of dw against V = left
  if (d_right) METIS_TRY(launch_factor_grad<true>(s, dw, dw_dtype, lddw, m, n, w->k, lq, nullptr, w->sigma, d_right, nullptr));
  return METIS_OK;
}

struct Side {
  const metis_nvfp4_t* res;   // residual, K-major along the contraction axis
  const metis_nvfp4_t* fc;    // factor along the contraction axis (k x K)
  const metis_nvfp4_t* fo;    // factor along the output axis      (k x M or k x N)
  const float* sigma;
  int k;
};

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

metis_status_t check_nvfp4(const metis_nvfp4_t* t) {
  if (!t || !t->codes || !t->scales || !t->tensor_scale) return METIS_ERR_INVALID_ARG;
  if (t->sf_layout != METIS_SF_TILED) return METIS_ERR_INVALID_ARG;
  if (t->k_len % 64 || t->rows <= 0) return METIS_ERR_SHAPE;
  return METIS_OK;
}

// Where the intermediates of one product live inside the caller's workspace.
struct Plan {
  int64_t M, N, K;
  int ka, kb, kc, kx;
  bool fuse;
  float *pm, *lcat, *rcat, *y0;
  __nv_bfloat16 *lx, *rx;
  size_t bytes;
};

metis_status_t make_plan(const Side& a, const Side& b, void* ws, size_t ws_bytes, Plan* pl) {
  METIS_TRY(check_nvfp4(a.res));
  METIS_TRY(check_nvfp4(b.res));
  pl->M = a.res->rows; pl->N = b.res->rows; pl->K = a.res->k_len;
  if (b.res->k_len != pl->K) return METIS_ERR_SHAPE;
  pl->ka = a.k; pl->kb = b.k; pl->kc = a.k + b.k; pl->bytes = 0;
  if (pl->kc == 0) return METIS_OK;
  const int64_t M = pl->M, N = pl->N, K = pl->K;
  const int ka = a.k, kb = b.k, kc = pl->kc;
  if (ka > LW_MAXK || kb > LW_MAXK) return METIS_ERR_SHAPE;
  if (ka) { METIS_TRY(check_nvfp4(a.fc)); METIS_TRY(check_nvfp4(a.fo)); if (a.fc->k_len != K || a.fo->k_len != M || !a.sigma) return METIS_ERR_SHAPE; }
  if (kb) { METIS_TRY(check_nvfp4(b.fc)); METIS_TRY(check_nvfp4(b.fo)); if (b.fc->k_len != K || b.fo->k_len != N || !b.sigma) return METIS_ERR_SHAPE; }
  unsigned char* w = reinterpret_cast<unsigned char*>(ws);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off += align256(bytes); return o; };
  pl->fuse = metis_gemm_tc_can_fuse(a.res, b.res);
  if (!pl->fuse && kc > 128) return METIS_ERR_SHAPE;    // layers below 256 rows hold the update operands in shared memory
  pl->kx = (2 * kc + 63) / 64 * 64;          // two BF16 column groups per rank-k term (see lowrank_finish_kernel)
  const size_t o_pm = take(sizeof(float) * (size_t)(ka * kb > 64 * 64 ? ka * kb : 64 * 64)), o_l = take(sizeof(float) * M * kc), o_r = take(sizeof(float) * N * kc);
  const size_t o_lx = pl->fuse ? take(sizeof(__nv_bfloat16) * M * pl->kx) : 0, o_rx = pl->fuse ? take(sizeof(__nv_bfloat16) * N * pl->kx) : 0;
  const size_t o_y0 = pl->fuse ? 0 : take(sizeof(float) * M * N);
  pl->bytes = off;
  if (!ws || off > ws_bytes) return METIS_ERR_WORKSPACE;
  pl->pm = reinterpret_cast<float*>(w + o_pm); pl->lcat = reinterpret_cast<float*>(w + o_l); pl->rcat = reinterpret_cast<float*>(w + o_r);
  pl->lx = pl->fuse ? reinterpret_cast<__nv_bfloat16*>(w + o_lx) : nullptr;
  pl->rx = pl->fuse ? reinterpret_cast<__nv_bfloat16*>(w + o_rx) : nullptr;
  pl->y0 = pl->fuse ? nullptr : reinterpret_cast<float*>(w + o_y0);
  return METIS_OK;
}

// Everything of one or two products that comes before their large GEMMs: the skinny products (straight into their slots of the concatenated
// operands; of a layer with fewer than 256 rows the residual product too) in one launch and the finishing kernels.
metis_status_t split_gemm_prologue(metis_context* ctx, const Side* const* a, const Side* const* b, const Plan* const* pl, int n, cudaStream_t s) {
  metis_gemm_job jobs[8], large[4];
  FinishArgs f[2] = {};
  int n_jobs = 0, n_large = 0, n_f = 0;
  bool wide = false, fused = false;
  int64_t mx[2] = {0, 0}, m_max = 0;
  int kx = 0, kb_max = 0, k_max = 0;
  for (int i = 0; i < n; ++i) {
    if (pl[i]->kc == 0) continue;
    const Side &sa = *a[i], &sb = *b[i];
    const Plan& p = *pl[i];
    const int ka = p.ka, kb = p.kb, kc = p.kc;
    if (!p.fuse) {
      if (metis_ceil_div(p.M, 128) * metis_ceil_div(p.N, 64) <= ctx->sm_count) jobs[n_jobs++] = {sa.res, sb.res, p.y0, p.N, false};
      else METIS_TRY(metis_launch_gemm_tc(ctx, sa.res, sb.res, p.y0, METIS_FP32, p.N, s));
    }
    // Rank 256, long and deep: 128 x 128 tiles read 140 bytes a cycle and SM, beyond what the L2 delivers, so such products keep the 256 x 256 tiles of the
    // two-CTA kernel, beside the group on the side stream or behind it.  Weight gradient of 16384 x 8192 x 8192: all in the group 664 us, so 641;
    // input and weight gradient 1492 and 1427; 16384 x 4096 x 14336 1318 and 1271.  With 4096 rows (half as many tiles as SMs) the group is the faster: 222
    // against 233 us at 16384 x 4096 x 4096; at K = 4096 they are equal.
    auto skinny = [&](const metis_nvfp4_t* r, const metis_nvfp4_t* fc, float* d) {
      const bool square = fc->rows >= 256 && r->rows >= 8192 && r->rows * r->k_len >= (int64_t)1 << 26;
      (square ? large[n_large++] : jobs[n_jobs++]) = {r, fc, d, kc, true};
    };
    if (kb) skinny(sa.res, sb.fc, p.lcat);
    if (ka) skinny(sb.res, sa.fc, p.rcat + kb);
    if (ka && kb) jobs[n_jobs++] = {sa.fc, sb.fc, p.pm, kb, true};
    FinishArgs& o = f[n_f];
    o.M = p.M; o.N = p.N; o.ka = ka; o.kb = kb; o.kx = p.kx;
    if (ka) { o.foa_codes = sa.fo->codes; o.foa_sf = sa.fo->scales; o.foa_layout = sa.fo->sf_layout; o.foa_ts = sa.fo->tensor_scale; }
    if (kb) { o.fob_codes = sb.fo->codes; o.fob_sf = sb.fo->scales; o.fob_layout = sb.fo->sf_layout; o.fob_ts = sb.fo->tensor_scale; }
    o.sa = sa.sigma; o.sb = sb.sigma; o.pm = p.pm; o.lcat = p.lcat; o.rcat = p.rcat; o.lx = p.lx; o.rx = p.rx;
    o.res_a_ts = sa.res->tensor_scale; o.res_b_ts = sb.res->tensor_scale;
    mx[n_f] = p.M > p.N ? p.M : p.N;
    if (p.M > m_max) m_max = p.M;
    wide |= ka > 64 || kb > 64; fused |= p.lx != nullptr;
    if (p.kx > kx) kx = p.kx;
    if (kb > kb_max) kb_max = kb;
    k_max = ka > k_max ? ka : k_max; k_max = kb > k_max ? kb : k_max;
    ++n_f;
  }
  if (n_f == 0) return METIS_OK;
  if (n_large) METIS_TRY(metis_fork(ctx, s, 1));           // (the group first: its CTAs are few and soon done)
  METIS_TRY(metis_launch_gemm_group(ctx, jobs, n_jobs, s));
  for (int i = 0; i < n_large; ++i)
    METIS_TRY(metis_launch_gemm_tc(ctx, large[i].a, large[i].b, large[i].d, METIS_FP32, large[i].ldd, i & 1 ? s : ctx->side[0]));
  if (n_large) METIS_TRY(metis_join(ctx, s, 0));
  const int64_t longest = mx[0] > mx[1] ? mx[0] : mx[1];
  if (wide) {
    METIS_CUDA_TRY(metis_launch_pdl(lowrank_deq_wide_kernel, dim3((unsigned)metis_ceil_div(longest, 32), (unsigned)n_f), dim3(256), 0, s, f[0], f[1])); METIS_COUNT_LAUNCH();
    if (kb_max) {                                           // (blocks of the rows of A alone: N may be beyond what a grid has in y)
      METIS_CUDA_TRY(metis_launch_pdl(lowrank_gemm_wide_kernel, dim3((unsigned)metis_ceil_div(kb_max, 64), (unsigned)metis_ceil_div(m_max, 64), (unsigned)n_f), dim3(256), 0, s,
                                      f[0], f[1])); METIS_COUNT_LAUNCH();
    }
    if (fused) {
      METIS_CUDA_TRY(metis_launch_pdl(lowrank_bf16_kernel, dim3((unsigned)metis_ceil_div(longest * (kx / 8), 256), (unsigned)n_f), dim3(256), 0, s, f[0], f[1])); METIS_COUNT_LAUNCH();
    }
    return METIS_OK;
  }
  // rows per warp: one while all rows together are not more than eight warps for every scheduler
  const int64_t rows = mx[0] + mx[1], per = 32ll * ctx->sm_count;
#define METIS_FINISH_J(R, J) METIS_CUDA_TRY(metis_launch_pdl((lowrank_finish_kernel<R, J>), dim3((unsigned)(n_first + metis_ceil_div(mx[1], 8 * (R)))), dim3(256), 0, s, f[0], f[1], (int)n_first))
#define METIS_FINISH(R) { const int64_t n_first = metis_ceil_div(mx[0], 8 * (R)); if (k_max <= 32) METIS_FINISH_J(R, 1); else METIS_FINISH_J(R, 2); METIS_COUNT_LAUNCH(); }
  if (rows <= per + per / 2) METIS_FINISH(1)
  else if (rows <= 3 * per) METIS_FINISH(2)
  else METIS_FINISH(4)
#undef METIS_FINISH_J
#undef METIS_FINISH
  return METIS_OK;
}

metis_status_t split_gemm_main(metis_context* ctx, const Side& a, const Side& b, const Plan& pl, void* d, int d_dtype, int64_t ldd,
                               cudaStream_t s) {
  if (pl.kc == 0) return metis_launch_gemm_tc(ctx, a.res, b.res, d, d_dtype, ldd, s);
  if (pl.fuse) {
    // residual x residual product and the rank-(ka+kb) correction accumulate into one FP32 tile in tensor memory
    return metis_launch_gemm_tc_fused(ctx, a.res, b.res, d, d_dtype, ldd, pl.lx, pl.rx, pl.kx, s);
  }
  dim3 grid((unsigned)metis_ceil_div(pl.N, 64), (unsigned)metis_ceil_div(pl.M, 64));
  const size_t smem = sizeof(float) * 2 * pl.kc * 68;
  METIS_CUDA_TRY(metis_launch_pdl(rank_update_kernel, grid, dim3(256), smem, s, (const float*)pl.y0, pl.M, pl.N, pl.kc, (const float*)pl.lcat, (const float*)pl.rcat, d, d_dtype, ldd)); METIS_COUNT_LAUNCH();
  return METIS_OK;
}

metis_status_t split_gemm(metis_context* ctx, const Side& a, const Side& b, void* d, int d_dtype, int64_t ldd, void* ws,
                          size_t ws_bytes, cudaStream_t s) {
  Plan pl;
  METIS_TRY(make_plan(a, b, ws, ws_bytes, &pl));
  const Side *pa = &a, *pb = &b;
  const Plan* pp = &pl;
  METIS_TRY(split_gemm_prologue(ctx, &pa, &pb, &pp, 1, s));
  return split_gemm_main(ctx, a, b, pl, d, d_dtype, ldd, s);
}

}  // namespace

metis_status_t metis_linear_set_attrs() {
  METIS_CUDA_TRY(cudaFuncSetAttribute(rank_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(sizeof(float) * 2 * 128 * 68)));
#define METIS_FG_ATTR(NT, TR, T, V) METIS_CUDA_TRY(cudaFuncSetAttribute(factor_grad_kernel<NT, TR, T, V>, cudaFuncAttributeMaxDynamicSharedMemorySize, fg_smem(NT, sizeof(T), 1 << 20)))
#define METIS_FG_ATTRS(NT) \
  METIS_FG_ATTR(NT, false, float, true); METIS_FG_ATTR(NT, false, float, false); METIS_FG_ATTR(NT, true, float, true); METIS_FG_ATTR(NT, true, float, false); \
  METIS_FG_ATTR(NT, false, __nv_bfloat16, true); METIS_FG_ATTR(NT, false, __nv_bfloat16, false); METIS_FG_ATTR(NT, true, __nv_bfloat16, true); \
  METIS_FG_ATTR(NT, true, __nv_bfloat16, false)
  METIS_FG_ATTRS(1); METIS_FG_ATTRS(2); METIS_FG_ATTRS(4); METIS_FG_ATTRS(6); METIS_FG_ATTRS(8);
#undef METIS_FG_ATTRS
#undef METIS_FG_ATTR
  return METIS_OK;
}

size_t metis_linear_ws_bytes(int64_t M, int64_t N, int k) {
  const int kc = 2 * k;
  const int kx = (2 * kc + 63) / 64 * 64;
  // sized for either path: FP32 staging of the main product (small shapes) or the BF16 correction operands
  const size_t pm_elems = (size_t)k * k > 64 * 64 ? (size_t)k * k : 64 * 64;
  return align256(sizeof(float) * M * N) + align256(sizeof(float) * pm_elems) +
         align256(sizeof(float) * M * (kc ? kc : 1)) + align256(sizeof(float) * N * (kc ? kc : 1)) +
         align256(sizeof(__nv_bfloat16) * M * (kx ? kx : 1)) + align256(sizeof(__nv_bfloat16) * N * (kx ? kx : 1)) +
         align256(sizeof(float) * (size_t)(k > 64 ? k : 64) * (size_t)metis_ceil_div(M > N ? M : N, FG_ROWS));     // partials of the sigma gradient
}

metis_status_t metis_linear_fwd(metis_handle_t h, const metis_operand_t* x, const metis_operand_t* w, void* y,
                                int32_t y_dtype, int64_t ldy, void* ws, size_t ws_bytes, metis_stream_t stream) {
  METIS_NVTX("metis_linear_fwd");
  if (!h || !x || !w || !y) return METIS_ERR_INVALID_ARG;
  if (y_dtype != METIS_BF16 && y_dtype != METIS_FP32) return METIS_ERR_INVALID_ARG;
  if (x->cols != w->cols || ldy < w->rows) return METIS_ERR_SHAPE;
  // contraction over in-features: X (l x m) by columns, W_t (n x m) by columns
  Side a{&x->res_by_cols, &x->right_q, &x->left_q, x->sigma, x->k};
  Side b{&w->res_by_cols, &w->right_q, &w->left_q, w->sigma, w->k};
  return split_gemm(h, a, b, y, y_dtype, ldy, ws, ws_bytes, reinterpret_cast<cudaStream_t>(stream));
}

metis_status_t metis_linear_bwd(metis_handle_t h, const metis_operand_t* dy, const metis_operand_t* x,
                                const metis_operand_t* w, void* dx, int32_t dx_dtype, int64_t lddx, void* dw,
                                int32_t dw_dtype, int64_t lddw, float* d_left, float* d_sigma, float* d_right,
                                void* ws, size_t ws_bytes, metis_stream_t stream) {
  METIS_NVTX("metis_linear_bwd");
  if (!h || !dy) return METIS_ERR_INVALID_ARG;
  if ((d_left || d_sigma || d_right) && (!dw || !w)) return METIS_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // every host-detectable error is reported before anything is enqueued
  if (dx && (!w || dy->cols != w->rows)) return METIS_ERR_SHAPE;
  if (dw && (!x || dy->rows != x->rows)) return METIS_ERR_SHAPE;
  if (dx && ((dx_dtype != METIS_BF16 && dx_dtype != METIS_FP32))) return METIS_ERR_INVALID_ARG;
  if (dw && ((dw_dtype != METIS_BF16 && dw_dtype != METIS_FP32))) return METIS_ERR_INVALID_ARG;
  if (dx && lddx < w->cols) return METIS_ERR_SHAPE;
  if (dw && lddw < x->cols) return METIS_ERR_SHAPE;
  if (dw && (d_left || d_sigma || d_right)) {
    if (w->rows != dy->cols || w->cols != x->cols) return METIS_ERR_SHAPE;
    METIS_TRY(factor_grads_check(w, d_left, d_sigma, ws, ws_bytes));
  }
  // dX (l x m) = D W_t, contraction over out-features n: D by columns, W_t by rows (stored m x n)
  Side da{&dy->res_by_cols, &dy->right_q, &dy->left_q, dy->sigma, dy->k};
  Side db = w ? Side{&w->res_by_rows, &w->left_q, &w->right_q, w->sigma, w->k} : Side{};
  // dW_t (n x m) = D^T X, contraction over tokens l: both by rows (stored n x l and m x l)
  Side wa{&dy->res_by_rows, &dy->left_q, &dy->right_q, dy->sigma, dy->k};
  Side wb = x ? Side{&x->res_by_rows, &x->left_q, &x->right_q, x->sigma, x->k} : Side{};
  if (dx && dw) {
    // Both products: with room for two sets of intermediates, everything that precedes the large GEMMs goes together.
    Plan pd, pw;
    METIS_TRY(make_plan(da, db, ws, ws_bytes, &pd));
    const size_t off = pd.bytes;
    const metis_status_t st = make_plan(wa, wb, ws ? reinterpret_cast<unsigned char*>(ws) + off : nullptr,
                                        ws_bytes > off ? ws_bytes - off : 0, &pw);
    if (st == METIS_OK) {
      const Side *as[2] = {&da, &wa}, *bs[2] = {&db, &wb};
      const Plan* ps[2] = {&pd, &pw};
      METIS_TRY(split_gemm_prologue(h, as, bs, ps, 2, s));
      METIS_TRY(split_gemm_main(h, da, db, pd, dx, dx_dtype, lddx, s));
      METIS_TRY(split_gemm_main(h, wa, wb, pw, dw, dw_dtype, lddw, s));
    } else if (st == METIS_ERR_WORKSPACE) {
      METIS_TRY(split_gemm(h, da, db, dx, dx_dtype, lddx, ws, ws_bytes, s));
      METIS_TRY(split_gemm(h, wa, wb, dw, dw_dtype, lddw, ws, ws_bytes, s));
    } else {
      return st;
    }
  } else if (dx) {
    METIS_TRY(split_gemm(h, da, db, dx, dx_dtype, lddx, ws, ws_bytes, s));
  } else if (dw) {
    METIS_TRY(split_gemm(h, wa, wb, dw, dw_dtype, lddw, ws, ws_bytes, s));
  }
  if (dw && (d_left || d_sigma || d_right))
    METIS_TRY(factor_grads(h, dw, dw_dtype, lddw, w, d_left, d_sigma, d_right, ws, ws_bytes, s));
  return METIS_OK;
}
