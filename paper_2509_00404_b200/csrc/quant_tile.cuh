// NVFP4 encoding of blocks of 16 values in registers (Section 2.3).  Used by the stand-alone quantizer and by the fused
// residual -> quantizer kernel of the split, so both produce identical codes for identical values.
#pragma once
#include "common.cuh"

namespace metis_qt {

constexpr int TILE = 128;
constexpr int THREADS = 256;

struct QuantParams {
  int64_t rows, cols;                 // source matrix extent
  int rounding;
  uint64_t seed;
  uint32_t stream_id;
  int64_t e_stride_r, e_stride_c;     // logical element index = r*e_stride_r + c*e_stride_c (keys the SR draw)
  // outputs (either may be absent: codes == nullptr)
  uint8_t* c_codes; uint8_t* c_scales; int c_layout;    // blocks along columns: stored rows x cols
  uint8_t* r_codes; uint8_t* r_scales; int r_layout;    // blocks along rows:    stored cols x rows
  // debug build: extents of the scale buffers (the code buffers hold rows * cols / 2 bytes) and the status word
  int64_t c_sf_bytes, r_sf_bytes;
  uint32_t* dbg;
  uint32_t* status;                   // set to METIS_DEV_NONFINITE where the tensor scale's amax is not finite (may be nullptr)
  PhiloxKeys keys;                    // round keys of `seed` (filled where the element draws are made in bulk)
};

// amax of the tensor about to be quantized is not a finite number (one thread of a launch calls)
__device__ __forceinline__ void check_amax(const QuantParams& p, const float* amax) {
  if (p.status != nullptr && !(fabsf(*amax) <= 3.0e38f)) atomicOr(p.status, METIS_DEV_NONFINITE);
}

// Encodes one block of 16 values; returns the scale byte, writes 8 code bytes.
__device__ __forceinline__ uint32_t encode_block(const float (&v)[16], const uint32_t (&u)[16], bool sr, float s_T,
                                                 float six_s_T, uint32_t (&packed)[2]) {
  // maximum by a tree: four dependent steps instead of sixteen
  float m8[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) m8[i] = fmaxf(fabsf(v[i]), fabsf(v[i + 8]));
  const float amax = fmaxf(fmaxf(fmaxf(m8[0], m8[4]), fmaxf(m8[1], m8[5])), fmaxf(fmaxf(m8[2], m8[6]), fmaxf(m8[3], m8[7])));
  float t = fminf(__fdiv_rn(amax, six_s_T), 448.0f);
  float sb;
  const uint32_t byte = metis_e4m3_ceil(t, &sb);
  const float r = sb == 0.0f ? 0.0f : __fdiv_rn(1.0f, __fmul_rn(sb, s_T));
  packed[0] = packed[1] = 0u;
  if (!sr) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t b = metis_e2m1x2_rne(__fmul_rn(v[2 * i], r), __fmul_rn(v[2 * i + 1], r));
      packed[i >> 2] |= b << (8 * (i & 3));
    }
  } else {
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const uint32_t c = metis_e2m1_sr(__fmul_rn(v[i], r), u[i]);
      packed[i >> 3] |= c << (4 * (i & 7));
    }
  }
  return byte;
}

// The element multiplier r = 1 / (E4M3(byte) * s_T) depends only on the block's scale byte and the tensor scale, so a
// kernel can evaluate the defined operations once per byte and look the result up per block (0 for byte 0).
constexpr int R_TABLE = 128;
__device__ __forceinline__ void fill_r_table(float* tab, float s_T, int tid, int nthreads) {
  for (int b = tid; b < R_TABLE; b += nthreads)
    tab[b] = (b == 0 || b == 127) ? 0.0f : __fdiv_rn(1.0f, __fmul_rn(metis_e4m3_value((uint32_t)b), s_T));
}

// four round-to-nearest-even code bytes (eight values) packed into one word
__device__ __forceinline__ uint32_t e2m1x8_rne(float a0, float a1, float a2, float a3, float a4, float a5, float a6, float a7) {
  uint32_t w;
  asm("{ .reg .b8 t0, t1, t2, t3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t0, %2, %1;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t1, %4, %3;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t2, %6, %5;\n"
      "cvt.rn.satfinite.e2m1x2.f32 t3, %8, %7;\n"
      "mov.b32 %0, {t0, t1, t2, t3}; }"
      : "=r"(w) : "f"(a0), "f"(a1), "f"(a2), "f"(a3), "f"(a4), "f"(a5), "f"(a6), "f"(a7));
  return w;
}

// What a 16-bit draw u contributes to the rounding of its element, one byte permutation of a Philox word that holds the draw in its
// low (hi = false) or high half:  256 u - 2^24 of the word as it is, or (COMPL) (65535 - u) 256 + 255 of its complement.
template <bool COMPL> constexpr uint32_t SR_SEL_LO = COMPL ? 0x5104u : 0x4105u;  // byte selectors, against 0xFF
template <bool COMPL> constexpr uint32_t SR_SEL_HI = COMPL ? 0x5324u : 0x4325u;
template <bool COMPL>
__device__ __forceinline__ uint32_t sr_term(uint32_t word, bool hi) { return __byte_perm(word, 0xFFu, hi ? SR_SEL_HI<COMPL> : SR_SEL_LO<COMPL>); }

// Eight stochastically rounded codes in one word; term[i] = sr_term of draw i.  The same decision as metis_e2m1_sr,
// arranged for the instruction mix of the SM (integer logic, shifts and compares issue at half the FP32 / IMAD rate, and bound
// this code):
//   b = max(a, RU(a/2 + 1/2)) maps a < 1 onto [1/2, 1] (the E2M1 grid {0, 1/2, 1} becomes {1/2, 3/4, 1}: one
//       mantissa bit per binade like the values from 1 up) and leaves a >= 1 alone, without a select;
//   with S = 4 bits(b) + (65535 - u) 256 + 255 the 22 mantissa bits below the grid bit carry into it exactly when  frac * 65536 > u
//       (4 frac22 + (65535 - u) 256 + 255 >= 2^24  <=>  frac22 > 64 u): comparison, selection and increment in one multiply-add.  Either S is
//       formed (COMPL) or its complement, ~S = term - 4 bits(b), where the draw enters as it is: complementing the Philox words costs half an
//       instruction per element, which the quantizer saves; the residual pass, at its 96 registers a thread, spills then
//       (8192 x 14336, k = 32, on a slower part: 214 us with S, 227 with ~S);
//   the magnitude code is bits 24 .. 26 of S, minus 4 modulo 8: the top bytes of four elements are gathered by byte permutations, the
//       two words of even and odd elements are merged and the complement and the eight "- 4" taken off together;
//   the sign nibbles are gathered with one funnel shift per element and masked once per word.
// (Against a compare per element with the draw shifted up and codes packed one by one: residual_tc_kernel 236 -> 204 us at 8192 x 14336, k = 32, the
// minimum per element below included, 199 us with the scale byte without branches; quantize_kernel 472 -> 371 us at 16384 x 14336 with
// both orientations, its third CTA per SM included, 340 us with the complement formed here, that scale byte and one block of code per loop.)
template <bool COMPL>
__device__ __forceinline__ uint32_t e2m1x8_sr(const float (&y)[8], const uint32_t (&term)[8]) {
  uint32_t s[8], sgn = 0u;
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    const float a = fabsf(y[i]);                           // at most 6 (the caller has seen to it)
    const uint32_t b4 = __float_as_uint(fmaxf(a, __fmaf_ru(a, 0.5f, 0.5f))) * 4u;
    s[i] = COMPL ? b4 + term[i] : term[i] - b4;
    sgn = __funnelshift_l(__float_as_uint(y[i]), sgn, 4);  // top nibble of y (sign and three exponent bits) shifted in
  }
  const uint32_t even = __byte_perm(__byte_perm(s[0], s[2], 0x0073u), __byte_perm(s[4], s[6], 0x7300u), 0x7610u);
  const uint32_t odd = __byte_perm(__byte_perm(s[1], s[3], 0x0073u), __byte_perm(s[5], s[7], 0x7300u), 0x7610u);
  const uint32_t mag = ((even & 0x0F0F0F0Fu) | ((odd * 16u) & 0xF0F0F0F0u));
  return ((mag & 0x77777777u) ^ (COMPL ? 0x44444444u : 0x33333333u)) | (sgn & 0x88888888u);
}

// largest magnitude of a block: eight three-input maxima, which pass a NaN over or (KEEP_NAN) on
template <bool KEEP_NAN>
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  if (KEEP_NAN) asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  else asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
template <bool KEEP_NAN>
__device__ __forceinline__ float amax16(const float (&v)[16]) {
  float m[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) m[i] = max3<KEEP_NAN>(fabsf(v[3 * i]), fabsf(v[3 * i + 1]), fabsf(v[3 * i + 2]));
  const float lo = max3<KEEP_NAN>(m[0], m[1], m[2]), hi = max3<KEEP_NAN>(m[3], m[4], fabsf(v[15]));
  return max3<KEEP_NAN>(lo, hi, hi);
}

// the byte of metis_e4m3_ceil without its branches: 0 for zero and a NaN
__device__ __forceinline__ uint32_t e4m3_ceil_byte(float t) {
  const uint32_t normal = ((__float_as_uint(t) + 0xFFFFFu) >> 20) - (120u << 3), subnormal = __float2uint_ru(__fmul_rn(t, 512.0f));
  return t > 0.015625f ? normal : subnormal;
}

// encode_block with the multiplier looked up in a table filled by fill_r_table (same bytes as encode_block).
// term[i] = sr_term<COMPL> of draw i (only read with stochastic rounding).
template <bool COMPL>
__device__ __forceinline__ uint32_t encode_block_tab(const float (&v)[16], const uint32_t (&term)[16], bool sr, float six_s_T,
                                                     const float* r_tab, uint32_t (&packed)[2]) {
  if (!sr) {
    const uint32_t byte = e4m3_ceil_byte(fminf(__fdiv_rn(amax16<false>(v), six_s_T), 448.0f));
    const float r = r_tab[byte];
    packed[0] = e2m1x8_rne(__fmul_rn(v[0], r), __fmul_rn(v[1], r), __fmul_rn(v[2], r), __fmul_rn(v[3], r),
                           __fmul_rn(v[4], r), __fmul_rn(v[5], r), __fmul_rn(v[6], r), __fmul_rn(v[7], r));
    packed[1] = e2m1x8_rne(__fmul_rn(v[8], r), __fmul_rn(v[9], r), __fmul_rn(v[10], r), __fmul_rn(v[11], r),
                           __fmul_rn(v[12], r), __fmul_rn(v[13], r), __fmul_rn(v[14], r), __fmul_rn(v[15], r));
    return byte;
  }
  float y0[8], y1[8];
  uint32_t t0[8], t1[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { t0[i] = term[i]; t1[i] = term[8 + i]; }
  const float amax = amax16<true>(v);
  uint32_t byte = e4m3_ceil_byte(fminf(__fdiv_rn(amax, six_s_T), 448.0f));
  float r = r_tab[byte];
  // values beyond 6 saturate, and a NaN is stored as 6.  They only occur where the block scale itself is saturated, the product
  // of the block maximum rounds up, or an element is a NaN, and the block maximum shows it, so the other blocks are spared a
  // minimum per element.  The scale of a block is that of its other elements (448 where there are none).
  if (__fmul_rn(amax, r) <= 6.0f) {
#pragma unroll
    for (int i = 0; i < 8; ++i) { y0[i] = __fmul_rn(v[i], r); y1[i] = __fmul_rn(v[8 + i], r); }
  } else {
    if (isnan(amax)) {
      byte = e4m3_ceil_byte(fminf(__fdiv_rn(amax16<false>(v), six_s_T), 448.0f));
      r = r_tab[byte];
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float a = __fmul_rn(v[i], r), b = __fmul_rn(v[8 + i], r);
      y0[i] = copysignf(fminf(fabsf(a), 6.0f), a); y1[i] = copysignf(fminf(fabsf(b), 6.0f), b);
    }
  }
  packed[0] = e2m1x8_sr<COMPL>(y0, t0);
  packed[1] = e2m1x8_sr<COMPL>(y1, t1);
  return byte;
}

}  // namespace metis_qt
