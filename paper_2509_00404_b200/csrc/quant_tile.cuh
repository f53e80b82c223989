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

// The scale byte of a block: the smallest E4M3 value not below t = min(amax / six, 448), the quotient rounded to nearest.
// six is the same for all blocks, so its reciprocal is taken once and the quotient corrected twice with its exact remainder.  The first
// correction leaves it within one unit in the last place, the second, with a correctly rounded reciprocal, rounds it as a division does
// (Markstein, IBM J. Res. Dev. 34, 1990).  That holds while no remainder is subnormal: amax >= lo with 2^-70 <= six <= 2^100 and lo = six 2^-30
// keeps the last bit of every product above 2^-149.  Other blocks are divided (zero, a NaN, one far below the tensor's maximum); an infinity
// gives a NaN here, and the largest scale like there.
struct BlockScaler { float six, inv, lo; };
__device__ __forceinline__ BlockScaler block_scaler(float s_T) {
  BlockScaler q;
  q.six = __fmul_rn(6.0f, s_T);
  const bool usable = q.six >= 0x1p-70f && q.six <= 0x1p100f;
  q.inv = usable ? __frcp_rn(q.six) : 0.0f;
  q.lo = usable ? q.six * 0x1p-30f : __int_as_float(0x7F800000);
  return q;
}
// t 2^-120, rounded up, has E4M3's exponents as an FP32 number, its subnormals among FP32's: one addition rounds either kind up to E4M3
__device__ __forceinline__ uint32_t e4m3_ceil_byte(float t) { return (__float_as_uint(__fmul_ru(t, 0x1p-120f)) + 0xFFFFFu) >> 20; }
__device__ __forceinline__ uint32_t scale_byte(float amax, const BlockScaler& q) {
  float t;
  if (amax >= q.lo && q.inv != 0.0f) {
    t = __fmul_rn(amax, q.inv);
    t = __fmaf_rn(__fmaf_rn(-t, q.six, amax), q.inv, t);
    t = __fmaf_rn(__fmaf_rn(-t, q.six, amax), q.inv, t);
  } else {
    t = __fdiv_rn(amax, q.six);
  }
  return e4m3_ceil_byte(fminf(t, 448.0f));
}

// two products at once
__device__ __forceinline__ void mul2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{ .reg .b64 a, b, d;\n"
      "mov.b64 a, {%2, %3};\n"
      "mov.b64 b, {%4, %5};\n"
      "mul.rn.f32x2 d, a, b;\n"
      "mov.b64 {%0, %1}, d; }"
      : "=f"(d0), "=f"(d1) : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
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

// Stochastically rounded codes.  The same decision as metis_e2m1_sr, arranged for the instruction mix of the SM (integer logic, shifts and
// compares issue at half the FP32 / IMAD rate, and bound this code):
//   z = RU(a 2^-126), a = |y| <= 6, is an FP32 number with E2M1's exponents: a < 1 becomes subnormal, rounded up to 22 bits below
//       the grid's spacing of 1/2, and a >= 1 is only scaled.  The bits of z are then the code in units of 2^22, for every binade
//       alike: no select, no offset;
//   with S = 4 bits(z) + (65535 - u) 256 + 255 the 22 bits below the grid carry into the code exactly when  frac * 65536 > u
//       (4 frac22 + (65535 - u) 256 + 255 >= 2^24  <=>  frac22 > 64 u): comparison, selection and increment in one multiply-add, and the
//       top byte of S is the code.  Either S is formed (COMPL) or its complement, ~S = term - 4 bits(z), where the draw enters as it is:
//       complementing the Philox words costs half an instruction per element, which the quantizer saves (the residual pass, at its 96 registers
//       a thread, spills then);
//   the codes of eight elements are gathered by byte permutations, those of even and of odd elements, and merged in one multiply-add;
//   the sign nibbles are gathered with one funnel shift per element, or, from BF16 pairs, with half a permutation.
// 16384 x 14336 BF16 in both orientations: 472 us with a compare per element; 341 us with a < 1 mapped onto
// [1/2, 1] by max(a, RU(a/2 + 1/2)), four masks and shifts per word of codes and a division per block; 317 us so, 309 us with the maxima
// on BF16 pairs, 276 us (30.4 instructions) with whole tiles in a kernel of their own (quantize_kernel).
// Residual pass, 8192 x 14336, k = 32: 231 -> 219 us (226 uncomplemented); 16384 x 4096, k = 64: 149 -> 139 us.
constexpr float SR_SCALE = 0x1p-126f;
template <bool COMPL>
__device__ __forceinline__ uint32_t sr_sum(float z, uint32_t term) { return COMPL ? __float_as_uint(z) * 4u + term : term - __float_as_uint(z) * 4u; }
// s: sums of eight elements; sgn: their signs on the top bits of the nibbles, other bits are ignored
template <bool COMPL>
__device__ __forceinline__ uint32_t e2m1x8_gather(const uint32_t (&s)[8], uint32_t sgn) {
  const uint32_t even = __byte_perm(__byte_perm(s[0], s[2], 0x0073u), __byte_perm(s[4], s[6], 0x7300u), 0x7610u);
  const uint32_t odd = __byte_perm(__byte_perm(s[1], s[3], 0x0073u), __byte_perm(s[5], s[7], 0x7300u), 0x7610u);
  // bytes 0 .. 7, or 255 less that: F0 | 15 - c and, with the four ones shifted in, 16 (15 - c) | 15
  const uint32_t mag = COMPL ? even + odd * 16u : ~(even & (odd * 16u + 15u));
  return mag | (sgn & 0x88888888u);
}
template <bool COMPL>
__device__ __forceinline__ uint32_t e2m1x8_sr(const float (&y)[8], const uint32_t (&term)[8]) {
  uint32_t s[8], sgn = 0u;
#pragma unroll
  for (int i = 7; i >= 0; --i) {
    s[i] = sr_sum<COMPL>(__fmul_ru(fabsf(y[i]), SR_SCALE), term[i]);
    sgn = __funnelshift_l(__float_as_uint(y[i]), sgn, 4);  // top nibble of y (sign and three exponent bits) shifted in
  }
  return e2m1x8_gather<COMPL>(s, sgn);
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

// encode_block with the multiplier looked up in a table filled by fill_r_table (same bytes as encode_block).
// term[i] = sr_term<COMPL> of draw i (only read with stochastic rounding).
template <bool COMPL>
__device__ __forceinline__ uint32_t encode_block_tab(const float (&v)[16], const uint32_t (&term)[16], bool sr, const BlockScaler& q,
                                                     const float* r_tab, uint32_t (&packed)[2]) {
  if (!sr) {
    const uint32_t byte = scale_byte(amax16<false>(v), q);
    const float r = r_tab[byte];
    float y[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) mul2(y[2 * i], y[2 * i + 1], v[2 * i], v[2 * i + 1], r, r);
    packed[0] = e2m1x8_rne(y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[7]);
    packed[1] = e2m1x8_rne(y[8], y[9], y[10], y[11], y[12], y[13], y[14], y[15]);
    return byte;
  }
  float y0[8], y1[8];
  uint32_t t0[8], t1[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) { t0[i] = term[i]; t1[i] = term[8 + i]; }
  const float amax = amax16<true>(v);
  uint32_t byte = scale_byte(amax, q);
  float r = r_tab[byte];
  // values beyond 6 saturate, and a NaN is stored as 6.  They only occur where the block scale itself is saturated, the product
  // of the block maximum rounds up, or an element is a NaN, and the block maximum shows it, so the other blocks are spared a
  // minimum per element.  The scale of a block is that of its other elements (448 where there are none).
  if (__fmul_rn(amax, r) <= 6.0f) {
#pragma unroll
    for (int i = 0; i < 4; ++i) { mul2(y0[2 * i], y0[2 * i + 1], v[2 * i], v[2 * i + 1], r, r); mul2(y1[2 * i], y1[2 * i + 1], v[8 + 2 * i], v[9 + 2 * i], r, r); }
  } else {
    if (isnan(amax)) {
      byte = scale_byte(amax16<false>(v), q);
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

// ---- the same for BF16 values in packed words, two elements each (lo, hi) ----
// Against the form on single values: the sign is masked once per word, both multiplications are two at a time, the maximum is taken on the bit
// patterns of a pair (a NaN is above every number) and the signs come by permutation from the words.

// largest pattern of either half over N words, signs left out; a NaN passes on
template <int N>
__device__ __forceinline__ uint32_t max_words(const uint32_t (&w)[N]) {
  uint32_t m = w[0];
#pragma unroll
  for (int i = 1; i < N; ++i) asm("max.NaN.xorsign.abs.bf16x2 %0, %0, %1;" : "+r"(m) : "r"(w[i]));
  return m & 0x7FFF7FFFu;
}
// Sums of eight words' elements: lo[i], hi[i] of word i, scaled by r0 and r1.  `fits`: no product is above 6 or a NaN; else the products are
// clamped (a NaN to 6) and the signs of the words' elements whose product is a NaN cleared.
__device__ __forceinline__ void sr_words(uint32_t (&w)[8], const uint32_t (&draw)[8], float r0, float r1, bool fits, uint32_t (&lo)[8], uint32_t (&hi)[8]) {
  float z0[8], z1[8];
  if (fits) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t m = w[i] & 0x7FFF7FFFu;
      asm("{ .reg .b64 a, b, c, d;\n"
          "mov.b64 a, {%2, %3};\n"
          "mov.b64 b, {%4, %5};\n"
          "mov.b64 c, {%6, %6};\n"
          "mul.rn.f32x2 d, a, b;\n"
          "mul.rp.f32x2 d, d, c;\n"
          "mov.b64 {%0, %1}, d; }"
          : "=f"(z0[i]), "=f"(z1[i]) : "f"(__uint_as_float(m << 16)), "f"(__uint_as_float(m & 0xFFFF0000u)), "f"(r0), "f"(r1), "f"(SR_SCALE));
    }
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float a = __fmul_rn(__uint_as_float((w[i] << 16) & 0x7FFFFFFFu), r0), b = __fmul_rn(__uint_as_float(w[i] & 0x7FFF0000u), r1);
      if (isnan(a)) w[i] &= ~0x8000u;
      if (isnan(b)) w[i] &= ~0x80000000u;
      z0[i] = __fmul_ru(fminf(a, 6.0f), SR_SCALE);
      z1[i] = __fmul_ru(fminf(b, 6.0f), SR_SCALE);
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    lo[i] = sr_sum<false>(z0[i], sr_term<false>(draw[i], false));
    hi[i] = sr_sum<false>(z1[i], sr_term<false>(draw[i], true));
  }
}
// the scale byte of a block whose maximum is a NaN is that of its other elements (448 where there are none)
__device__ __forceinline__ uint32_t scale_byte_bf16(uint32_t pattern, const BlockScaler& q) { return scale_byte(__uint_as_float(pattern << 16), q); }
__device__ __forceinline__ float max_no_nan(float m, uint32_t pattern) { return fmaxf(m, fabsf(__uint_as_float(pattern << 16))); }

// a block of 16 in eight words
__device__ __forceinline__ uint32_t encode_words_sr(uint32_t (&w)[8], const uint32_t (&draw)[8], const BlockScaler& q, const float* r_tab, uint32_t (&packed)[2]) {
  const uint32_t m2 = max_words(w), m = max(m2 & 0xFFFFu, m2 >> 16);
  uint32_t byte = scale_byte_bf16(m, q);
  float r = r_tab[byte];
  const bool fits = __fmul_rn(__uint_as_float(m << 16), r) <= 6.0f;
  if (!fits && m > 0x7F80u) {
    float o = __int_as_float(0x7FC00000);
#pragma unroll
    for (int i = 0; i < 8; ++i) o = max_no_nan(max_no_nan(o, w[i] & 0xFFFFu), w[i] >> 16);
    byte = scale_byte(o, q);
    r = r_tab[byte];
  }
  uint32_t lo[8], hi[8];
  sr_words(w, draw, r, r, fits, lo, hi);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t s[8] = {lo[4 * h], hi[4 * h], lo[4 * h + 1], hi[4 * h + 1], lo[4 * h + 2], hi[4 * h + 2], lo[4 * h + 3], hi[4 * h + 3]};
    const uint32_t a = __byte_perm(w[4 * h], w[4 * h + 1], 0x7351u), b = __byte_perm(w[4 * h + 2], w[4 * h + 3], 0x7351u);   // top bytes: lo, lo, hi, hi
    const uint32_t e = __byte_perm(a, b, 0x5410u) >> 4, o = __byte_perm(a, b, 0x7632u);
    packed[h] = e2m1x8_gather<false>(s, (e & 0x0F0F0F0Fu) | (o & 0xF0F0F0F0u));
  }
  return byte;
}

// two blocks side by side, of the lo and of the hi elements of 16 words; the draws' words stand 64 words apart
__device__ __forceinline__ void encode_columns_sr(uint32_t (&w)[16], const uint32_t* draws, const BlockScaler& q, const float* r_tab, uint32_t& byte0, uint32_t& byte1,
                                                  uint32_t (&p0)[2], uint32_t (&p1)[2]) {
  const uint32_t m = max_words(w), m0 = m & 0xFFFFu, m1 = m >> 16;
  byte0 = scale_byte_bf16(m0, q); byte1 = scale_byte_bf16(m1, q);
  float r0 = r_tab[byte0], r1 = r_tab[byte1];
  const bool fits = __fmul_rn(__uint_as_float(m0 << 16), r0) <= 6.0f && __fmul_rn(__uint_as_float(m1 << 16), r1) <= 6.0f;
  if (!fits && (m0 > 0x7F80u || m1 > 0x7F80u)) {
    float o0 = __int_as_float(0x7FC00000), o1 = o0;
#pragma unroll
    for (int i = 0; i < 16; ++i) { o0 = max_no_nan(o0, w[i] & 0xFFFFu); o1 = max_no_nan(o1, w[i] >> 16); }
    byte0 = scale_byte(o0, q); byte1 = scale_byte(o1, q);
    r0 = r_tab[byte0]; r1 = r_tab[byte1];
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t wh[8], draw[8], s0[8], s1[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) { wh[i] = w[8 * h + i]; draw[i] = draws[(8 * h + i) * 64]; }
    sr_words(wh, draw, r0, r1, fits, s0, s1);
    const uint32_t a = __byte_perm(wh[0], wh[2], 0x7351u), b = __byte_perm(wh[4], wh[6], 0x7351u);     // top bytes: lo, lo, hi, hi
    const uint32_t c = __byte_perm(wh[1], wh[3], 0x7351u), d = __byte_perm(wh[5], wh[7], 0x7351u);
    const uint32_t e0 = __byte_perm(a, b, 0x5410u) >> 4, o0 = __byte_perm(c, d, 0x5410u), e1 = __byte_perm(a, b, 0x7632u) >> 4, o1 = __byte_perm(c, d, 0x7632u);
    p0[h] = e2m1x8_gather<false>(s0, (e0 & 0x0F0F0F0Fu) | (o0 & 0xF0F0F0F0u));
    p1[h] = e2m1x8_gather<false>(s1, (e1 & 0x0F0F0F0Fu) | (o1 & 0xF0F0F0F0u));
  }
}

}  // namespace metis_qt
