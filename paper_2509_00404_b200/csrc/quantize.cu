// Tensor amax and the stand-alone NVFP4 quantizer (Section 2.3; value set of Appendix C.1).
#include <type_traits>

#include "quant_tile.cuh"

namespace {

// amax|x| of a strided matrix: one read of the tensor, bound by HBM.  A unit of work is UNROLL 16-byte vectors per
// thread, all requested before the first is looked at; `tpr` threads (a power of two, at most 256) stand side by side on a row,
// so that narrow rows do not idle the block, and one 32-bit division per unit finds the unit's place (a 64-bit division per
// vector and scalar FP32 loads held the kernel at 3.6 TB/s for BF16 and 1.1 TB/s for FP32).  Units are walked
// from the end of the tensor to its start: the quantizer that follows reads from the start, which is then what L2 holds.
// STREAM: a tensor well beyond the L2 is loaded evict-first, so that what the L2 holds of others is not written back or lost for lines nobody finds
// again (16384 x 14336 BF16: 83 -> 69 us, the quantizer behind it as before).
template <int DTYPE, bool STREAM>
__global__ void __launch_bounds__(256)
amax_kernel(const void* __restrict__ x, int64_t rows, int64_t cols, int64_t ld, int tpr, int narrow, uint32_t segs, uint32_t units, float* __restrict__ out) {
  // |x| as a bit pattern: non-negative floats order like their bit patterns, infinity above every number and a
  // NaN above infinity, so a non-finite element survives the reduction (fmaxf would drop a NaN)
  metis_pdl_wait();
  constexpr int UNROLL = 8;
  constexpr int E = DTYPE == METIS_BF16 ? 8 : 4;           // elements per load
  uint32_t m = 0u;
  const int tx = threadIdx.x & (tpr - 1), ty = threadIdx.x / tpr, rpp = 256 / tpr;
  const int64_t vecs = cols / E;
  for (uint32_t i = blockIdx.x; i < units; i += gridDim.x) {
    const uint32_t u = units - 1 - i, rg = u / segs, sg = u - rg * segs;
    const int64_t r0 = (int64_t)rg * rpp * (narrow ? UNROLL : 1) + ty, c0 = (int64_t)sg * tpr * UNROLL + tx;
    uint4 q[UNROLL];
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
      // rows of at most tpr vectors: the unit is UNROLL row groups; longer rows: UNROLL steps along the row
      const int64_t r = narrow ? r0 + (int64_t)j * rpp : r0, c = narrow ? c0 : c0 + (int64_t)j * tpr;
      q[j] = make_uint4(0u, 0u, 0u, 0u);
      if (r < rows && c < vecs) {
        const uint4* at = reinterpret_cast<const uint4*>(reinterpret_cast<const unsigned char*>(x) + (r * ld + c * E) * (16 / E));
        q[j] = STREAM ? __ldcs(at) : __ldg(at);
      }
    }
#pragma unroll
    for (int j = 0; j < UNROLL; ++j) {
      const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (DTYPE == METIS_BF16) { m = max(m, (w[e] << 16) & 0x7FFFFFFFu); m = max(m, w[e] & 0x7FFF0000u); }
        else m = max(m, w[e] & 0x7FFFFFFFu);
      }
    }
  }
  // The launch of the quantizer behind this kernel overlaps its end.  (At the head, the quantizer's CTAs, which need the result for
  // all they do, would stand on SMs for as long as this kernel runs: up to 67 us, out of the reach of other streams.)
  metis_pdl_trigger();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  __shared__ uint32_t wmax[8];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, wmax[w]);
    atomicMax(reinterpret_cast<unsigned int*>(out), m);
  }
}

// two draws in a word: those of elements e and e + step
__device__ __noinline__ uint32_t draw_pair(uint64_t e, uint64_t step, uint64_t seed, uint32_t stream) {
  return metis_draw_u16(e, seed, stream) | (metis_draw_u16(e + step, seed, stream) << 16);
}

// Stand-alone quantizer, 128 x 128 elements per CTA.
//  pass 1  every thread loads 16 consecutive elements of a row (32 bytes of BF16) - exactly one block along the
//          columns - and, if that orientation is wanted, encodes it in registers and writes its 8 code bytes
//          straight to global memory (8 threads = 64 contiguous bytes of a row); the values (BF16 or FP32) and
//          the stochastic-rounding draws go to shared memory for pass 2
//  pass 2  blocks along the rows: a thread reads 16 values down a column from shared memory, encodes them and
//          stages the bytes; the transposed codes and both scale tiles are then written out coalesced
constexpr int QK_CP = metis_qt::TILE / 2 + 8;                     // pitch of a staged row of row-block codes, bytes
// T = __nv_bfloat16 or float: element type of the shared tile (= input type).  WHOLE: every tile lies in the matrix, rows start on 32-byte boundaries,
// scales are tiled and draws are numbered along the rows, so that a block has no bounds, no second form of load, draw or scale and nothing to clear:
// with these decisions in its loops the kernel executed 34.9 instructions per element, 31.7 without, and they are what bounds it
// (70 % of the issue slots, 70 % of the integer pipe).  A grid of resident CTAs that walks the tiles changed neither count nor time.
template <typename T, bool SR, bool WHOLE>
__global__ void __launch_bounds__(metis_qt::THREADS, sizeof(T) == 4 ? (SR ? 2 : 3) : (SR ? 3 : 4))    // as many CTAs as their shared memory allows
quantize_kernel(const T* __restrict__ x, int64_t ld, metis_qt::QuantParams p, const float* __restrict__ tscale_src,
                int tscale_is_amax, float* ts_out0, float* ts_out1) {
  using namespace metis_qt;
  // Shared-memory layouts, chosen so that every access of a warp touches each bank once.
  //   BF16 tile and draws: rows of 256 bytes = 16 chunks of 16 bytes, chunk ch stored at ch ^ (ch >> 3): the eight
  //     lanes of a quarter warp store the even (or odd) chunks of one row, which the swizzle spreads over all banks;
  //     pass 2 reads 32 consecutive words of a row, a permutation of the chunks inside one 128-byte window.
  //   FP32 tile: rows of 512 bytes = 32 chunks of 16 bytes, chunk ch stored at ch ^ (ch >> 3): the eight lanes of a quarter warp store
  //     every fourth chunk of a row onto all banks; pass 2 reads 32 consecutive columns, a permutation inside one 128-byte window.
  //     (Element stores into rows of 129 words met four to a bank; with them and unpipelined loads: 100 us at 14336 x 4096, 73 us so.)
  //   staged row-block codes: 72-byte rows; a BF16 thread owns two adjacent columns, so column c is staged in row
  //     (c >> 1) + 64 (c & 1) and the 32 lanes of a store write 32 consecutive rows (18 words apart: 16 lanes cover
  //     the 32 banks with their 8 bytes each).
  constexpr int TP = TILE;                                       // tile pitch in elements
  extern __shared__ __align__(16) unsigned char smem[];
  T* tile = reinterpret_cast<T*>(smem);                                        // [TILE][TP]
  uint8_t* codes_s = smem + sizeof(T) * TILE * TP;                             // [TILE][QK_CP] row-block codes
  // [TILE][8] scales of the column blocks, written out before pass 2 puts those of the row blocks in their place: with
  // an area for each, two CTAs of the stochastic-rounding kernel fitted an SM instead of three
  uint8_t* sfc = codes_s + TILE * QK_CP;
  uint8_t* sfr = sfc;
  float* r_tab = reinterpret_cast<float*>(sfc + TILE * 8);                     // multiplier per scale byte
  uint16_t* rnd = reinterpret_cast<uint16_t*>(r_tab + R_TABLE);                // [TILE][TILE] draws (SR only)

  auto staged_row = [](int c) { return sizeof(T) == 2 ? (c >> 1) + 64 * (c & 1) : c; };
  // Scale bytes of the tile, from their staging area [stored row][8] to global memory.  The four blocks of a 64-element
  // K group are adjacent in both layouts, so they go out as one word per thread (256 words per tile and orientation;
  // in the tiled layout consecutive threads write consecutive words of a 512-byte atom, and blocks or rows of the atom
  // that lie outside the matrix are its zero padding); an unaligned linear layout takes the byte path.
  auto write_scales = [&](uint8_t* dst, int64_t extent, int layout, int64_t bpr, const uint8_t* src, bool staged, int v_rows, int v_k, int64_t g_row0, int64_t g_blk0) {
    (void)extent;
    const bool tiled = WHOLE || layout == METIS_SF_TILED;
    if (WHOLE || ((tiled || (bpr & 3) == 0) && (reinterpret_cast<uintptr_t>(dst) & 3) == 0)) {
      const int i = threadIdx.x;                                          // THREADS == 2 * TILE words
      const int atom = tiled ? i >> 7 : i & 1;
      const int r = tiled ? ((i & 127) >> 2) + 32 * (i & 3) : i >> 1;
      if (WHOLE || (atom * 64 < v_k && (r < v_rows || tiled))) {
        const uint32_t w = WHOLE || r < v_rows ? *reinterpret_cast<const uint32_t*>(src + (staged ? staged_row(r) : r) * 8 + atom * 4) : 0u;
        // a tile starts on a 128-row slab and a 128-element K group: metis_sf_offset(g_row0 + r, g_blk0 + 4 atom) in parts
        const int64_t off = tiled ? ((g_row0 >> 7) * (bpr >> 2) + (g_blk0 >> 2)) * 512 + i * 4 : (g_row0 * bpr + g_blk0) + (r * bpr + atom * 4);
        METIS_DBG_GUARD(p.dbg, off, 4, extent) *reinterpret_cast<uint32_t*>(dst + off) = w;
      }
    } else {
      for (int i = threadIdx.x; i < TILE * 8; i += THREADS) {
        int r, b;
        if (tiled) { const int atom = i >> 9, w = i & 511; r = (w >> 4) + 32 * ((w >> 2) & 3); b = atom * 4 + (w & 3); }
        else { r = i >> 3; b = i & 7; }
        if (b * 16 < v_k && (r < v_rows || tiled))
          METIS_DBG_GUARD(p.dbg, metis_sf_offset(g_row0 + r, g_blk0 + b, bpr, layout), 1, extent) dst[metis_sf_offset(g_row0 + r, g_blk0 + b, bpr, layout)] = r < v_rows ? src[(staged ? staged_row(r) : r) * 8 + b] : (uint8_t)0;
      }
    }
  };
  const int tid = threadIdx.x;
  metis_pdl_wait();
  const int64_t row0 = (int64_t)blockIdx.y * TILE, col0 = (int64_t)blockIdx.x * TILE;
  const float s_T = tscale_is_amax ? metis_tensor_scale(*tscale_src) : *tscale_src;
  const BlockScaler scaler = block_scaler(s_T);
  if (blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) {
    if (ts_out0 != nullptr && ts_out0 != tscale_src) *ts_out0 = s_T;
    if (ts_out1 != nullptr && ts_out1 != tscale_src) *ts_out1 = s_T;
    if (tscale_is_amax) check_amax(p, tscale_src);
  }
  constexpr bool sr = SR;
  fill_r_table(r_tab, s_T, tid, THREADS);
  const bool want_c = p.c_codes != nullptr, want_r = p.r_codes != nullptr;
  const int vrows = WHOLE ? TILE : (int)min((int64_t)TILE, p.rows - row0), vcols = WHOLE ? TILE : (int)min((int64_t)TILE, p.cols - col0);
  const bool fast_draws = WHOLE || (p.e_stride_c == 1 && (p.e_stride_r & 7) == 0);
  const bool wide_ld = WHOLE || sizeof(T) == 2 && (ld & 15) == 0 && (reinterpret_cast<uintptr_t>(x) & 31) == 0;   // 32-byte aligned blocks

  // ---- pass 1 ----
  // BF16, round to nearest: all global loads of the tile are issued before the first block is encoded, 128 bytes per thread in flight.
  // BF16, stochastic: bound by instructions, a block ahead is enough, and a loop of two blocks instead of four side by side keeps the code in
  // the instruction cache (16384 x 14336, both orientations: one block 283 us, two 276, four 286)
  constexpr int AHEAD = SR ? 1 : 4;
  uint4 raw[sizeof(T) == 2 ? 2 * AHEAD : 1];
  const int b = tid & 7, r0 = tid >> 3;                    // this thread's blocks: (r0 + 32 it, b)
  const T* src0 = x + (row0 + r0) * ld + col0 + b * 16;
  auto load_bf16 = [&](int it) {
    uint4& lo = raw[sizeof(T) == 2 ? 2 * (it % AHEAD) : 0];
    uint4& hi = raw[sizeof(T) == 2 ? 2 * (it % AHEAD) + 1 : 0];
    if (!WHOLE) lo = hi = make_uint4(0u, 0u, 0u, 0u);
    if (WHOLE || (r0 + 32 * it < vrows && b * 16 < vcols)) {
      const uint4* src = reinterpret_cast<const uint4*>(src0 + (int64_t)(32 * it) * ld);
      if (wide_ld) {                                       // one 32-byte load per block: consecutive lanes, consecutive 32 bytes
        asm volatile("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(lo.x), "=r"(lo.y), "=r"(lo.z), "=r"(lo.w), "=r"(hi.x), "=r"(hi.y), "=r"(hi.z), "=r"(hi.w)
                     : "l"(src));
      } else {
        lo = src[0]; hi = src[1];
      }
    }
  };
  if (sizeof(T) == 2) {
#pragma unroll
    for (int it = 0; it < AHEAD; ++it) load_bf16(it);
  }
  // FP32: the block of the next round is loaded while this round's is encoded
  float4 nxt[sizeof(T) == 4 ? 4 : 1];
  auto load_fp32 = [&](int it) {
    const bool in = WHOLE || (r0 + 32 * it < vrows && b * 16 < vcols);
    const float4* src = reinterpret_cast<const float4*>(src0 + (int64_t)(32 * it) * ld);
#pragma unroll
    for (int j = 0; j < 4; ++j) nxt[sizeof(T) == 4 ? j : 0] = in ? src[j] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  };
  if (sizeof(T) == 4) load_fp32(0);
  __syncthreads();                                         // multiplier table complete (the tile loads are in flight)
  const int64_t gc = col0 + b * 16;
  int64_t code_at = (row0 + r0) * (p.cols / 2) + gc / 2;   // of the block's codes; the next block is 32 rows on
  uint64_t draw_at = ((uint64_t)(row0 + r0) * (uint64_t)p.e_stride_r + (uint64_t)gc) >> 3;
#pragma unroll (SR ? 2 : 4)
  for (int it = 0; it < 4; ++it) {
    const int r = r0 + 32 * it;
    const bool in = WHOLE || (r < vrows && b * 16 < vcols);
    float v[16];
    uint32_t u[16], w[8];
    if (sizeof(T) == 2) {
      const uint4 q0 = raw[sizeof(T) == 2 ? 2 * (it % AHEAD) : 0], q1 = raw[sizeof(T) == 2 ? 2 * (it % AHEAD) + 1 : 0];
      if (SR && it < 3) load_bf16(it + 1);
      w[0] = q0.x; w[1] = q0.y; w[2] = q0.z; w[3] = q0.w; w[4] = q1.x; w[5] = q1.y; w[6] = q1.z; w[7] = q1.w;
#pragma unroll
      for (int j = 0; j < 8; ++j) { v[2 * j] = __uint_as_float(w[j] << 16); v[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u); }
      if (want_r) {
        uint4* trow = reinterpret_cast<uint4*>(smem + r * 256);
        trow[(2 * b) ^ (b >> 2)] = q0;
        trow[(2 * b + 1) ^ (b >> 2)] = q1;
      }
    } else {
      float4 q[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) { q[j] = nxt[sizeof(T) == 4 ? j : 0]; v[4 * j] = q[j].x; v[4 * j + 1] = q[j].y; v[4 * j + 2] = q[j].z; v[4 * j + 3] = q[j].w; }
      if (it < 3) load_fp32(it + 1);
      if (want_r) {
        float4* trow = reinterpret_cast<float4*>(smem + r * 512);
#pragma unroll
        for (int j = 0; j < 4; ++j) trow[(4 * b + j) ^ (b >> 1)] = q[j];
      }
    }
    uint32_t nw[8];                                        // draws, two per word
    if (sr) {
      if (fast_draws) {
        const uint4 w0 = metis_philox_block_keys(draw_at, p.keys, p.stream_id), w1 = metis_philox_block_keys(draw_at + 1, p.keys, p.stream_id);
        nw[0] = w0.x; nw[1] = w0.y; nw[2] = w0.z; nw[3] = w0.w; nw[4] = w1.x; nw[5] = w1.y; nw[6] = w1.z; nw[7] = w1.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          nw[j] = draw_pair((uint64_t)(row0 + r) * (uint64_t)p.e_stride_r + (uint64_t)(gc + 2 * j) * (uint64_t)p.e_stride_c, (uint64_t)p.e_stride_c, p.seed, p.stream_id);
      }
      draw_at += 4 * (uint64_t)p.e_stride_r;               // 32 rows, eight draws to a Philox block
#pragma unroll
      for (int j = 0; j < 8; ++j) { u[2 * j] = sr_term<false>(nw[j], false); u[2 * j + 1] = sr_term<false>(nw[j], true); }
      if (want_r) {
        if (sizeof(T) == 2) {
          uint4* drow = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(rnd) + r * 256);
          drow[(2 * b) ^ (b >> 2)] = make_uint4(nw[0], nw[1], nw[2], nw[3]);
          drow[(2 * b + 1) ^ (b >> 2)] = make_uint4(nw[4], nw[5], nw[6], nw[7]);
        } else {
          uint32_t* dst = reinterpret_cast<uint32_t*>(rnd + r * TILE + b * 16);
#pragma unroll
          for (int j = 0; j < 8; ++j) dst[j] = nw[j];
        }
      }
    }
    if (want_c) {
      uint32_t packed[2];
      const uint32_t byte = SR && sizeof(T) == 2 ? encode_words_sr(w, nw, scaler, r_tab, packed) : encode_block_tab<false>(v, u, sr, scaler, r_tab, packed);
      if (in) METIS_DBG_GUARD(p.dbg, code_at, 8, p.rows * p.cols / 2) *reinterpret_cast<uint2*>(p.c_codes + code_at) = make_uint2(packed[0], packed[1]);
      code_at += 16 * p.cols;
      sfc[r * 8 + b] = in ? (uint8_t)byte : (uint8_t)0;
    }
  }
  __syncthreads();
  if (want_c) write_scales(p.c_scales, p.c_sf_bytes, p.c_layout, p.cols / 16, sfc, false, vrows, vcols, row0, col0 / 16);
  // ---- pass 2 ----
  if (want_r) {
    __syncthreads();                                       // the column blocks' scales have been read
    if (sizeof(T) == 2) {
      // BF16 tile: a thread takes two adjacent columns (one 32-bit shared load per row) and four of the eight
      // row blocks, i.e. eight blocks in two rounds of four
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        const int wd = tid & 63, b = (tid >> 6) + 4 * it;         // columns 2 wd, 2 wd + 1: word wd of a tile row
        const int pw = ((((wd >> 2) ^ (wd >> 5)) << 2) | (wd & 3));    // its swizzled position
        uint32_t p0[2], p1[2], byte0, byte1;
        const uint32_t* col = reinterpret_cast<const uint32_t*>(smem) + b * 16 * 64 + pw;
        if constexpr (SR) {
          const uint32_t* dcol = reinterpret_cast<const uint32_t*>(rnd) + b * 16 * 64 + pw;
          uint32_t w[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) w[i] = col[i * 64];
          encode_columns_sr(w, dcol, scaler, r_tab, byte0, byte1, p0, p1);
        } else {
          float v0[16], v1[16];
          const uint32_t none[16] = {};
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const uint32_t w = col[i * 64];
            v0[i] = __uint_as_float(w << 16); v1[i] = __uint_as_float(w & 0xFFFF0000u);
          }
          byte0 = encode_block_tab<false>(v0, none, false, scaler, r_tab, p0);
          byte1 = encode_block_tab<false>(v1, none, false, scaler, r_tab, p1);
        }
        *reinterpret_cast<uint2*>(codes_s + wd * QK_CP + b * 8) = make_uint2(p0[0], p0[1]);
        sfr[wd * 8 + b] = (uint8_t)byte0;
        *reinterpret_cast<uint2*>(codes_s + (64 + wd) * QK_CP + b * 8) = make_uint2(p1[0], p1[1]);
        sfr[(64 + wd) * 8 + b] = (uint8_t)byte1;
      }
    } else {
#pragma unroll 1
    for (int it = 0; it < 4; ++it) {
      const int c = tid & 127, b = (tid >> 7) + 2 * it;
      float v[16];
      uint32_t u[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) v[i] = reinterpret_cast<const float*>(tile)[(b * 16 + i) * TP + (((c >> 2) ^ (c >> 5)) << 2 | (c & 3))];
      if (sr) {
#pragma unroll
        for (int i = 0; i < 16; ++i) u[i] = sr_term<false>((uint32_t)rnd[(b * 16 + i) * TILE + c], false);
      }
      uint32_t packed[2];
      const uint32_t byte = encode_block_tab<false>(v, u, sr, scaler, r_tab, packed);
      *reinterpret_cast<uint2*>(codes_s + c * QK_CP + b * 8) = make_uint2(packed[0], packed[1]);
      sfr[c * 8 + b] = (uint8_t)byte;
    }
    }
    __syncthreads();
    int64_t at = (col0 + r0) * (p.rows / 2) + row0 / 2 + b * 8;               // columns r0, r0 + 32, ...
    const uint8_t* from = codes_s + staged_row(r0) * QK_CP + b * 8;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
      if (WHOLE || (r0 + 32 * it < vcols && b * 16 < vrows))
        METIS_DBG_GUARD(p.dbg, at, 8, p.rows * p.cols / 2) *reinterpret_cast<uint2*>(p.r_codes + at) = *reinterpret_cast<const uint2*>(from + (sizeof(T) == 2 ? 16 : 32) * it * QK_CP);
      at += 16 * p.rows;
    }
    write_scales(p.r_scales, p.r_sf_bytes, p.r_layout, p.rows / 16, sfr, true, vcols, vrows, col0, row0 / 16);
  }
}

template <typename T>
constexpr size_t quantize_smem(bool sr) {
  return sizeof(T) * metis_qt::TILE * metis_qt::TILE + metis_qt::TILE * QK_CP +
         metis_qt::TILE * 8 + sizeof(float) * metis_qt::R_TABLE + (sr ? sizeof(uint16_t) * metis_qt::TILE * metis_qt::TILE : 0);
}

}  // namespace

metis_status_t metis_quantize_set_attrs() {
  using namespace metis_qt;
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<__nv_bfloat16, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<__nv_bfloat16>(true)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<__nv_bfloat16, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<__nv_bfloat16>(true)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<float, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<float>(true)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<float, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<float>(true)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<__nv_bfloat16, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<__nv_bfloat16>(false)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<__nv_bfloat16, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<__nv_bfloat16>(false)));
  METIS_CUDA_TRY(cudaFuncSetAttribute(quantize_kernel<float, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)quantize_smem<float>(false)));
  return METIS_OK;
}

constexpr int64_t METIS_L2_BYTES = 126ll << 20;

metis_status_t metis_launch_amax(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, float* amax_out,
                                 cudaStream_t s, bool zeroed) {
  const bool bf = dtype == METIS_BF16;
  const int64_t e = bf ? 8 : 4;
  // the quantizer behind it wants the same of the operand: whole 16-byte loads
  if (cols % e || ld % e || !metis_aligned16(x)) return METIS_ERR_ALIGNMENT;
  if (!zeroed) METIS_CUDA_TRY(cudaMemsetAsync(amax_out, 0, sizeof(float), s));
  if (rows * cols == 0) return METIS_OK;
  if (ld == cols) { cols = rows * cols; rows = 1; ld = cols; }                  // contiguous: one long row
  const int64_t vecs = cols / e;
  int tpr = 256;
  while (tpr > 1 && tpr / 2 >= vecs) tpr /= 2;
  const bool narrow = vecs <= tpr;                                              // rows of at most one step of the block
  // Longer rows: a unit is 8 tpr vectors of each of 256 / tpr rows, and what lies beyond a row's end or the last row is not loaded.  Of at least 32
  // threads a row (512 bytes side by side) the count that makes the fewest units, the largest of equals.
  auto units_of = [&](int t) { return metis_ceil_div(rows, 256 / t) * metis_ceil_div(vecs, (int64_t)t * 8); };
  if (!narrow)
    for (int t = 128; t >= 32; t /= 2)
      if (units_of(t) < units_of(tpr)) tpr = t;
  const int64_t segs = narrow ? 1 : metis_ceil_div(vecs, (int64_t)tpr * 8);
  const int64_t groups = metis_ceil_div(rows, (int64_t)(256 / tpr) * (narrow ? 8 : 1));
  const int64_t units = groups * segs;
  if (units > 0xFFFFFFFFll) return METIS_ERR_SHAPE;
  // Resident CTAs that walk the units (one reduction and one atomic each) up to 5/4 of the L2 (8192 x 4160 FP32, 136 MB: 66.1 us, streamed 66.4).  Beyond a CTA per unit: 12 and 13 units a CTA
  // left an eighth of the last round idle (16384 x 14336 BF16, with its quantizer: 224 -> 214 us, evict-first 208; 16384 x 8192 134 -> 123; of
  // tensors that fit, 4160 x 2752 FP32 29.0 -> 29.1, evict-first 32.2: the quantizer finds less).
  const bool stream = rows * cols * (bf ? 2 : 4) > METIS_L2_BYTES / 4 * 5 && units <= 0x7FFFFFFFll;
  const unsigned grid = (unsigned)(stream || units < 148 * 8 ? units : 148 * 8);
  auto launch = [&](auto kernel) { return metis_launch_pdl(kernel, dim3(grid), dim3(256), (size_t)0, s, x, rows, cols, ld, tpr, narrow ? 1 : 0, (uint32_t)segs, (uint32_t)units, amax_out); };
  if (bf) METIS_CUDA_TRY(stream ? launch(amax_kernel<METIS_BF16, true>) : launch(amax_kernel<METIS_BF16, false>));
  else METIS_CUDA_TRY(stream ? launch(amax_kernel<METIS_FP32, true>) : launch(amax_kernel<METIS_FP32, false>));
  METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  return METIS_OK;
}


// Few long rows (the transposed split factors: k x len FP32, blocks along the contiguous dimension only): one
// thread per block of 16, no tiles, no shared memory.  Threads beyond `rows` inside the last 128-row slab of the
// tiled scale layout write zero scale bytes.
__device__ __forceinline__ void rowblocks_body(const float* x, int64_t ld, const metis_qt::QuantParams& p,
                                               const float* __restrict__ tscale_src, int tscale_is_amax, float* ts_out,
                                               const unsigned long long* __restrict__ keys, float* flip) {
  const int64_t bpr = p.cols / 16;
  const int64_t rows_pad = p.c_layout == METIS_SF_TILED ? (p.rows + 127) / 128 * 128 : p.rows;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= rows_pad * bpr) return;
  const int64_t r = idx / bpr, b = idx % bpr;
  if (r >= p.rows) { p.c_scales[metis_sf_offset(r, b, bpr, p.c_layout)] = 0; return; }
  const float s_T = tscale_is_amax ? metis_tensor_scale(*tscale_src) : *tscale_src;
  if (idx == 0 && ts_out != nullptr) *ts_out = s_T;
  const bool sr = p.rounding == METIS_ROUND_SR;
  float v[16];
  uint32_t u[16];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 q = *reinterpret_cast<const float4*>(x + r * ld + b * 16 + i * 4);
    v[4 * i] = q.x; v[4 * i + 1] = q.y; v[4 * i + 2] = q.z; v[4 * i + 3] = q.w;
  }
  if (keys != nullptr && (keys[r] & 1ull)) {               // the sign convention of the factor pair: this vector is flipped, in place
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = -v[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(flip + r * ld + b * 16 + i * 4) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
  }
  if (sr) {
    if (p.e_stride_c == 1 && (p.e_stride_r & 7) == 0) {
      const uint64_t e0 = (uint64_t)r * (uint64_t)p.e_stride_r + (uint64_t)b * 16u;
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const uint4 w = metis_philox_block((e0 >> 3) + h2, p.seed, p.stream_id);
#pragma unroll
        for (uint32_t hh = 0; hh < 8; ++hh) u[8 * h2 + hh] = metis_u16_of(w, hh);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        u[i] = metis_draw_u16((uint64_t)r * (uint64_t)p.e_stride_r + (uint64_t)(b * 16 + i) * (uint64_t)p.e_stride_c, p.seed, p.stream_id);
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) u[i] = 0u;
  }
  uint32_t packed[2];
  const uint32_t byte = metis_qt::encode_block(v, u, sr, s_T, __fmul_rn(6.0f, s_T), packed);
  *reinterpret_cast<uint2*>(p.c_codes + r * (p.cols / 2) + b * 8) = make_uint2(packed[0], packed[1]);
  p.c_scales[metis_sf_offset(r, b, bpr, p.c_layout)] = (uint8_t)byte;
}

__global__ void __launch_bounds__(256)
quantize_rowblocks_kernel(const float* __restrict__ x, int64_t ld, metis_qt::QuantParams p, const float* __restrict__ tscale_src,
                          int tscale_is_amax, float* ts_out) {
  metis_pdl_wait();
  if (tscale_is_amax && blockIdx.x == 0 && threadIdx.x == 0) metis_qt::check_amax(p, tscale_src);
  rowblocks_body(x, ld, p, tscale_src, tscale_is_amax, ts_out, nullptr, nullptr);
}

// ------------------------------------------------------------------------------------------------
// Comparison recipe of Section 4: random Hadamard transform of every 16-block along the columns, then NVFP4.
// y = H16 (s * x) / 4, four butterfly stages in binary32 (distance 1, 2, 4, 8; (a, b) -> (a + b, a - b)), signs
// s from bit 15 of the Philox draw of the column index (stream METIS_STREAM_SIGNS).
__device__ __forceinline__ void rht_block(const void* __restrict__ x, int dtype, int64_t ld, int64_t r, int64_t b, uint64_t seed, float (&v)[16]) {
  const uint4 w0 = metis_philox_block((uint64_t)b * 2, seed, METIS_STREAM_SIGNS), w1 = metis_philox_block((uint64_t)b * 2 + 1, seed, METIS_STREAM_SIGNS);
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const float xv = metis_ld_as_float(x, dtype, r * ld + b * 16 + i);
    const uint32_t u = metis_u16_of(i < 8 ? w0 : w1, (uint32_t)(i & 7));
    v[i] = (u & 0x8000u) ? -xv : xv;
  }
#pragma unroll
  for (int h = 1; h < 16; h <<= 1) {
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if ((i & h) == 0) { const float a = v[i], c = v[i + h]; v[i] = __fadd_rn(a, c); v[i + h] = __fsub_rn(a, c); }
  }
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __fmul_rn(v[i], 0.25f);
}

__global__ void __launch_bounds__(256)
rht_amax_kernel(const void* __restrict__ x, int dtype, int64_t rows, int64_t cols, int64_t ld, uint64_t seed, float* __restrict__ amax_out) {
  const int64_t bpr = cols / 16;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  uint32_t m = 0u;
  if (idx < rows * bpr) {
    float v[16];
    rht_block(x, dtype, ld, idx / bpr, idx % bpr, seed, v);
#pragma unroll
    for (int i = 0; i < 16; ++i) m = max(m, __float_as_uint(v[i]) & 0x7FFFFFFFu);      // ordered bit patterns: a NaN survives
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, o));
  if ((threadIdx.x & 31) == 0 && m) atomicMax(reinterpret_cast<unsigned int*>(amax_out), m);
}

__global__ void __launch_bounds__(256)
rht_quantize_kernel(const void* __restrict__ x, int dtype, int64_t ld, metis_qt::QuantParams p, const float* __restrict__ amax, float* ts_out) {
  const int64_t bpr = p.cols / 16;
  const int64_t rows_pad = p.c_layout == METIS_SF_TILED ? (p.rows + 127) / 128 * 128 : p.rows;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= rows_pad * bpr) return;
  const int64_t r = idx / bpr, b = idx % bpr;
  if (r >= p.rows) { p.c_scales[metis_sf_offset(r, b, bpr, p.c_layout)] = 0; return; }
  const float s_T = metis_tensor_scale(*amax);
  if (idx == 0) *ts_out = s_T;
  const bool sr = p.rounding == METIS_ROUND_SR;
  float v[16];
  uint32_t u[16];
  rht_block(x, dtype, ld, r, b, p.seed, v);
#pragma unroll
  for (int i = 0; i < 16; ++i) u[i] = 0u;
  if (sr) {
    const uint64_t e0 = (uint64_t)r * (uint64_t)p.cols + (uint64_t)b * 16u;
#pragma unroll
    for (int h2 = 0; h2 < 2; ++h2) {
      const uint4 w = metis_philox_block((e0 >> 3) + h2, p.seed, p.stream_id);
#pragma unroll
      for (uint32_t hh = 0; hh < 8; ++hh) u[8 * h2 + hh] = metis_u16_of(w, hh);
    }
  }
  uint32_t packed[2];
  const uint32_t byte = metis_qt::encode_block(v, u, sr, s_T, __fmul_rn(6.0f, s_T), packed);
  *reinterpret_cast<uint2*>(p.c_codes + r * (p.cols / 2) + b * 8) = make_uint2(packed[0], packed[1]);
  p.c_scales[metis_sf_offset(r, b, bpr, p.c_layout)] = (uint8_t)byte;
}

metis_status_t metis_launch_quantize_rht(metis_context* ctx, const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, int rounding, uint64_t seed,
                                         uint32_t stream_id, const metis_nvfp4_t* out, float* amax_ws, cudaStream_t s) {
  using namespace metis_qt;
  QuantParams p{};
  p.rows = rows; p.cols = cols; p.rounding = rounding; p.seed = seed; p.stream_id = stream_id; p.e_stride_r = cols; p.e_stride_c = 1;
  p.c_codes = out->codes; p.c_scales = out->scales; p.c_layout = out->sf_layout;
  METIS_CUDA_TRY(cudaMemsetAsync(amax_ws, 0, sizeof(float), s));
  const int64_t bpr = cols / 16;
  rht_amax_kernel<<<(unsigned)metis_ceil_div(rows * bpr, 256), 256, 0, s>>>(x, dtype, rows, cols, ld, seed, amax_ws); METIS_COUNT_LAUNCH();
  METIS_TRY(metis_launch_amax_check(ctx, amax_ws, s));
  const int64_t rows_pad = p.c_layout == METIS_SF_TILED ? (rows + 127) / 128 * 128 : rows;
  rht_quantize_kernel<<<(unsigned)metis_ceil_div(rows_pad * bpr, 256), 256, 0, s>>>(x, dtype, ld, p, amax_ws, out->tensor_scale); METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  return METIS_OK;
}

// two factor tensors in one launch (blockIdx.y selects): the left and right factors of a decomposition
// (keys: the sign keys of the vectors, or nullptr; x is then flipped where the key says so)
struct RowblocksJob { float* x; int64_t ld; metis_qt::QuantParams p; const float* tscale_src; float* ts_out; const unsigned long long* keys; };
__global__ void __launch_bounds__(256)
quantize_rowblocks_pair_kernel(RowblocksJob a, RowblocksJob b, metis_split_checks checks) {
  const RowblocksJob& j = blockIdx.y == 0 ? a : b;
  metis_pdl_wait();
  if (checks.status != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 32) {
    // device-detected conditions of the split that these factors belong to (amax is kept as an ordered bit pattern, so a NaN ranks above every number)
    uint32_t bits = 0u;
    if (threadIdx.x == 0 && !(fabsf(*checks.amax) <= 3.0e38f)) bits |= METIS_DEV_NONFINITE;
    for (int i = threadIdx.x; i < checks.k; i += 32)
      if (!(fabs(checks.evals[i]) <= 1.0e300)) bits |= METIS_DEV_NUMERIC;
    if (bits) atomicOr(checks.status, bits);
  }
  rowblocks_body(j.x, j.ld, j.p, j.tscale_src, 1, j.ts_out, j.keys, j.x);
}

metis_status_t metis_launch_quantize(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, int rounding,
                                     uint64_t seed, uint32_t stream_id, int64_t e_stride_r, int64_t e_stride_c,
                                     const float* tscale_src, int tscale_is_amax, const metis_nvfp4_t* by_cols,
                                     const metis_nvfp4_t* by_rows, cudaStream_t s, uint32_t* dbg_status) {
  using namespace metis_qt;
  // (dbg_status: also told of an amax that is not finite)
  if (rows == 0 || cols == 0) return METIS_OK;
  // vector loads of 16 elements per thread: the rows must start on 16-byte boundaries
  if (cols % 16 || (dtype == METIS_BF16 ? ld % 8 : ld % 4)) return METIS_ERR_ALIGNMENT;
  QuantParams p{};
  p.rows = rows; p.cols = cols; p.rounding = rounding; p.seed = seed; p.stream_id = stream_id;
  p.e_stride_r = e_stride_r; p.e_stride_c = e_stride_c;
  p.keys = metis_philox_keys(seed);
  if (by_cols) { p.c_codes = by_cols->codes; p.c_scales = by_cols->scales; p.c_layout = by_cols->sf_layout; p.c_sf_bytes = (int64_t)metis_sf_bytes(rows, cols, p.c_layout); }
  if (by_rows) { p.r_codes = by_rows->codes; p.r_scales = by_rows->scales; p.r_layout = by_rows->sf_layout; p.r_sf_bytes = (int64_t)metis_sf_bytes(cols, rows, p.r_layout); }
  p.dbg = p.status = dbg_status;
  if (dtype == METIS_FP32 && by_cols && !by_rows && rows <= 64) {
    const int64_t rows_pad = p.c_layout == METIS_SF_TILED ? (rows + 127) / 128 * 128 : rows;
    METIS_CUDA_TRY(metis_launch_pdl(quantize_rowblocks_kernel, dim3((unsigned)metis_ceil_div(rows_pad * (cols / 16), 256)), dim3(256), (size_t)0, s,
                                    reinterpret_cast<const float*>(x), ld, p, tscale_src, tscale_is_amax, by_cols->tensor_scale)); METIS_COUNT_LAUNCH();
    return METIS_OK;
  }
  const bool sr = rounding == METIS_ROUND_SR;
  dim3 grid((unsigned)metis_ceil_div(cols, TILE), (unsigned)metis_ceil_div(rows, TILE));
  float* t0 = by_cols ? by_cols->tensor_scale : nullptr; float* t1 = by_rows ? by_rows->tensor_scale : nullptr;
  // whole tiles: 16384 x 14336 BF16, both orientations, stochastic 309 -> 276 us, to nearest 147 -> 137 us; 4096 x 4096
  // FP32 stochastic 31.9 -> 29.0 us.  FP32 to nearest is bound by its reads and was slower so (21.2 -> 22.3 us).  Other calls keep every check.
  const bool whole = rows % TILE == 0 && cols % TILE == 0 && e_stride_c == 1 && e_stride_r % 8 == 0 && ld % 16 == 0 && (reinterpret_cast<uintptr_t>(x) & 31) == 0 &&
                     (!by_cols || (p.c_layout == METIS_SF_TILED && (reinterpret_cast<uintptr_t>(p.c_scales) & 3) == 0)) &&
                     (!by_rows || (p.r_layout == METIS_SF_TILED && (reinterpret_cast<uintptr_t>(p.r_scales) & 3) == 0));
  auto launch = [&](auto kernel, auto xt) { return metis_launch_pdl(kernel, grid, dim3(THREADS), quantize_smem<std::remove_const_t<std::remove_pointer_t<decltype(xt)>>>(sr), s, xt, ld, p, tscale_src, tscale_is_amax, t0, t1); };
  auto pick = [&](auto xt) {
    using T = std::remove_const_t<std::remove_pointer_t<decltype(xt)>>;
    if (sr) return whole ? launch(quantize_kernel<T, true, true>, xt) : launch(quantize_kernel<T, true, false>, xt);
    if constexpr (sizeof(T) == 2) {
      if (whole) return launch(quantize_kernel<T, false, true>, xt);
    }
    return launch(quantize_kernel<T, false, false>, xt);
  };
  if (dtype == METIS_BF16) METIS_CUDA_TRY(pick(reinterpret_cast<const __nv_bfloat16*>(x)));
  else METIS_CUDA_TRY(pick(reinterpret_cast<const float*>(x)));
  METIS_COUNT_LAUNCH();
  METIS_CUDA_TRY(cudaGetLastError());
  return METIS_OK;
}

// The two FP32 factor tensors of a decomposition (k x rows and k x cols, k <= 64, blocks along the long dimension,
// tensor scale from each tensor's own amax) in one launch.
metis_status_t metis_launch_quantize_factors(float* left, int64_t rows, float* right, int64_t cols, int k, int rounding,
                                             uint64_t seed, const float* amax_left, const float* amax_right,
                                             const metis_nvfp4_t* lq, const metis_nvfp4_t* rq, cudaStream_t s, const unsigned long long* keys,
                                             const metis_split_checks* checks) {
  using namespace metis_qt;
  if (k <= 0 || k > 256 || rows % 16 || cols % 16) return METIS_ERR_SHAPE;
  RowblocksJob a{}, b{};
  a.keys = b.keys = keys;
  a.x = left; a.ld = rows; a.tscale_src = amax_left; a.ts_out = lq->tensor_scale;
  a.p.rows = k; a.p.cols = rows; a.p.rounding = rounding; a.p.seed = seed; a.p.stream_id = METIS_STREAM_LEFT;
  a.p.e_stride_r = rows; a.p.e_stride_c = 1; a.p.c_codes = lq->codes; a.p.c_scales = lq->scales; a.p.c_layout = lq->sf_layout;
  b.x = right; b.ld = cols; b.tscale_src = amax_right; b.ts_out = rq->tensor_scale;
  b.p.rows = k; b.p.cols = cols; b.p.rounding = rounding; b.p.seed = seed; b.p.stream_id = METIS_STREAM_RIGHT;
  b.p.e_stride_r = cols; b.p.e_stride_c = 1; b.p.c_codes = rq->codes; b.p.c_scales = rq->scales; b.p.c_layout = rq->sf_layout;
  const int64_t pad_a = a.p.c_layout == METIS_SF_TILED ? (k + 127) / 128 * 128 : k, pad_b = b.p.c_layout == METIS_SF_TILED ? (k + 127) / 128 * 128 : k;
  const int64_t work_a = pad_a * (rows / 16), work_b = pad_b * (cols / 16);
  const unsigned gx = (unsigned)metis_ceil_div(work_a > work_b ? work_a : work_b, 256);
  METIS_CUDA_TRY(metis_launch_pdl(quantize_rowblocks_pair_kernel, dim3(gx, 2), dim3(256), (size_t)0, s, a, b, checks != nullptr ? *checks : metis_split_checks{})); METIS_COUNT_LAUNCH();
  return METIS_OK;
}
