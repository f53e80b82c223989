// One-CTA dense linear algebra of a decomposition (n <= 72): FP64 Cholesky factorisation and the symmetric
// eigen-decomposition.  Both are latency chains on one SM, so what counts is the number of dependent steps and how long one is.
#pragma once
#include "common.cuh"

namespace metis_small {

constexpr int MAXQ = 72;                                // k + p at most (k = 64 with p = 8)
constexpr int PITCH = MAXQ + 4;                         // doubles; 4 or 12 mod 16: every fragment access below is conflict-free

// 1/sqrt(x) in FP64: scaled into the FP32 range by an even power of two, FP32 seed, two Newton steps
__device__ __forceinline__ double rsqrt64(double x) {
  int e;
  const double mant = frexp(x, &e);                     // x = mant * 2^e, mant in [0.5, 1)
  const int e2 = e & ~1;
  const double xs = ldexp(mant, e - e2);                // in [0.5, 2)
  double y = (double)rsqrtf((float)xs);
  y = y * (1.5 - 0.5 * xs * y * y);
  y = y * (1.5 - 0.5 * xs * y * y);
  return ldexp(y, -(e2 / 2));
}

// 1/x in FP64: the hardware's FP64 reciprocal seed (error below 2^-20) and two Newton steps
__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(y, fma(-x, y, 1.0), y);
  y = fma(y, fma(-x, y, 1.0), y);
  return y;
}

// FP64 tensor-core tile: d (8 x 8) += a (8 x 4) b (4 x 8).  Lane (g = lane / 4, q = lane % 4) holds a[g][q], b[q][g] and
// d[g][2q], d[g][2q + 1].
__device__ __forceinline__ void dmma(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};" : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// (row, column) of lower tile o, counted row by row
__device__ __forceinline__ void lower_tile(int o, int& ti, int& tj) {
  ti = (int)(0.5f * (sqrtf(8.0f * (float)o + 1.0f) - 1.0f));
  tj = o - ti * (ti + 1) / 2;
}

// In-place Cholesky factorisation of the lower triangle of Y (n x n, n8 = n rounded up to a multiple of eight, row pitch P doubles,
// rows and columns up to n8 must exist and be zero beyond n), called by all nthr >= n8 - 8 threads of the CTA.
// Panels of eight columns: every warp factorises the panel's diagonal block in registers (lane = row; a column step is one
// pivot broadcast, one reciprocal and one multiply-add deep, without a barrier) and carries 32 rows below it along; then all warps subtract
// the panel's rank-8 product from the trailing tiles on the FP64 tensor cores, two tiles at a time.  (One barrier per
// column with the matrix spread over 256 threads' registers took 800 cycles a column.)  A pivot not above `tol` marks a dependent column:
// it takes no part in the updates and ends as a zero column with inv_out[j] = 0; otherwise inv_out[j] = 1 / L[j][j].
// *dmin_out (optional): the smallest accepted pivot.
template <int P>
__device__ __forceinline__ void cta_cholesky(double* Y, int n, double tol, double* inv_out, double* dmin_out, int nthr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n_warps = nthr >> 5;
  const int n8 = (n + 7) & ~7, g = lane >> 2, q = lane & 3;
  double dmin = 1e300;
  for (int c0 = 0; c0 < n8; c0 += 8) {
    const int r = c0 + 8 + 32 * warp + lane, rd_ = c0 + (lane & 7);             // a row below the block, a row of the block
    double vd[8], inv = 0.0;
    const bool busy = warp == 0 || c0 + 8 + 32 * warp < n8;
    if (busy) {
      double v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) { vd[c] = Y[rd_ * P + c0 + c]; v[c] = r < n8 ? Y[r * P + c0 + c] : 0.0; }
      double my_pivot = 0.0;                            // lane j < 8: pivot of column c0 + j
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double d = __shfl_sync(0xFFFFFFFFu, vd[j], j);
        const double rd = d > tol ? rcp64(d) : 0.0;
        if ((lane & 7) == j) my_pivot = d;
        const double ld = vd[j] * rd, l = v[j] * rd;
#pragma unroll
        for (int c = j + 1; c < 8; ++c) {
          const double u = __shfl_sync(0xFFFFFFFFu, vd[j], c);
          vd[c] = fma(-ld, u, vd[c]);
          v[c] = fma(-l, u, v[c]);
        }
      }
      const bool ok = my_pivot > tol;
      inv = ok ? rsqrt64(my_pivot) : 0.0;
      if (ok) dmin = fmin(dmin, my_pivot);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const double ic = __shfl_sync(0xFFFFFFFFu, inv, c);
        vd[c] *= ic;
        if (r < n8) Y[r * P + c0 + c] = v[c] * ic;
      }
    }
    __syncthreads();                                    // the block has been read by every warp: its factor may be stored
    if (warp == 0 && lane < 8) {
      if (c0 + lane < n) inv_out[c0 + lane] = inv;
#pragma unroll
      for (int c = 0; c < 8; ++c) Y[rd_ * P + c0 + c] = c <= lane ? vd[c] : 0.0;
    }
    // trailing tiles (ti >= tj > panel): Y -= L_panel L_panel^T
    const int first = c0 / 8 + 1, nt = n8 / 8 - first, tiles = nt * (nt + 1) / 2;
    for (int o = warp; o < tiles; o += 2 * n_warps) {
      double acc[2][2], a[2][2], b[2][2];
      double* out[2];
      const bool two = o + n_warps < tiles;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        int ti, tj;
        lower_tile(u == 0 || !two ? o : o + n_warps, ti, tj);
        const int ri = 8 * (first + ti) + g, rj = 8 * (first + tj) + g;
        out[u] = Y + ri * P + 8 * (first + tj) + 2 * q;
        acc[u][0] = out[u][0]; acc[u][1] = out[u][1];
#pragma unroll
        for (int h = 0; h < 2; ++h) { a[u][h] = -Y[ri * P + c0 + 4 * h + q]; b[u][h] = Y[rj * P + c0 + 4 * h + q]; }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < 2; ++u) dmma(acc[u], a[u][h], b[u][h]);
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (u == 0 || two) { out[u][0] = acc[u][0]; out[u][1] = acc[u][1]; }
    }
    __syncthreads();
  }
  if (dmin_out != nullptr && warp == 0) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) dmin = fmin(dmin, __shfl_xor_sync(0xFFFFFFFFu, dmin, o));
    if (lane == 0) *dmin_out = dmin;
  }
  __syncthreads();
}

// X = L^-1 (nothing is written above the diagonal blocks) for the factor of cta_cholesky, by all nthr threads: the 8 x 8 diagonal
// blocks first (lane = column), then a warp per block column, X_ib = -X_ii sum_k L_ik X_kb on the FP64 tensor cores
// without a barrier.  inv: reciprocal pivots (zero for a dependent column, whose row of X is then zero).
template <int P>
__device__ __forceinline__ void cta_invert_lower(const double* L, const double* inv, int n, double* X, int xp, int nthr) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, q = lane & 3, nb = (n + 7) / 8;
  for (int b = warp; b < nb; b += nthr >> 5) {
    if (lane < 8) {
      double x[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < i; ++k) s = fma(L[(8 * b + i) * P + 8 * b + k], x[k], s);
        const double r = 8 * b + i < n ? inv[8 * b + i] : 0.0;
        x[i] = i == lane ? r : (i > lane ? -r * s : 0.0);
        X[(8 * b + i) * xp + 8 * b + lane] = x[i];
      }
    }
  }
  __syncthreads();
  for (int b = warp; b < nb; b += nthr >> 5) {
    for (int i = b + 1; i < nb; ++i) {
      double t[2][2] = {};
      for (int k = b; k < i; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h) dmma(t[h], L[(8 * i + g) * P + 8 * k + 4 * h + q], X[(8 * k + 4 * h + q) * xp + 8 * b + g]);
      double* out = X + (8 * i + g) * xp + 8 * b + 2 * q;
      out[0] = t[0][0] + t[1][0]; out[1] = t[0][1] + t[1][1];
      __syncwarp();
      double d[2] = {0.0, 0.0};
#pragma unroll
      for (int h = 0; h < 2; ++h) dmma(d, -X[(8 * i + g) * xp + 8 * i + 4 * h + q], X[(8 * i + 4 * h + q) * xp + 8 * b + g]);
      __syncwarp();
      out[0] = d[0]; out[1] = d[1];
      __syncwarp();
    }
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------------------------
// Symmetric positive semi-definite eigen-decomposition in one CTA.
//   1. the matrix, sorted by descending diagonal, is factorised G = L L^T (FP64; dependent columns zeroed);
//   2. one-sided Jacobi on the columns of L in FP32: Y = L J with orthogonal columns, so the normalised columns approximate the
//      eigenvectors.  Eight lanes own two blocks of two columns: one round loads four columns, forms their six inner
//      products at once, works out the four rotations between the blocks on the 4 x 4 Gram matrix in registers and
//      applies them - one barrier and one reduction for what takes two of each when single couples are rotated.  A round
//      is bound by latency and by its warps' own instruction streams (n = 40: 784 cycles; sixteen lanes a group: 990);
//   3. FP64 refinement of the eigenvectors U (Ogita and Aishima, "Iterative refinement for symmetric eigenvalue
//      decomposition", 2018): with R = I - U^T U and S = U^T G U, U += U E, E_ij = (S_ij + s_j R_ij) / (s_j - s_i), E_ii = R_ii / 2,
//      s_i = S_ii / (1 - R_ii); the error is squared by each step.  S is formed as W^T W with W = L^T U, which keeps the
//      relative accuracy of small eigenvalues.  The products run on the FP64 tensor cores;
//   4. eigenvalues too close to be separated this way (|E_ij| above 1/16, or E as a whole not small) send the matrix back to
//      step 2 with a tight exit test; if pairs are still open after that, they are only orthonormalised in step 3 and FP64
//      one-sided Jacobi sweeps on the columns of W = L^T U, U rotated along, finish the work (repeated eigenvalues).
// Precision: the columns of U leave the loop orthonormal, and the pairs of W orthogonal, to about 1e-12 (FP64 rotations
// with the exit test cos^2 < 1e-8, which this replaces, left 1e-9 ... 1e-12); FP32 only decides how good the start is.
// Input: Gram matrix (ld x ld, leading n x n block used).  Output: eigenvalues descending, eigenvectors as columns of
// evecs[n][n].
// Measured alone: n = 40 63 us for a sampled operand and 70 us for one decomposed from every row (seven sweeps), n = 32 32 us; about three
// quarters of it is the Jacobi phase.  The FP64 one-sided Jacobi before it took 113 - 126 us (n = 40), 52 us (n = 32), 250 us
// (n = 64) and 440 us (n = 72) inside a layer step, against 56 - 64, 31, 122 and 239 us.  Repeated eigenvalues, the worst case of
// step 4, are what got slower: 190 us at n = 40, half of them equal to the last digit; a decomposition of 1024 x 768 from every
// row, k = 32, all planted values equal, 333 -> 407 us.  (FP64 sweeps at once instead of the second attempt: 392 -> 494 us sampled.)
constexpr int EIG_THREADS = 512;
constexpr int EIG_MAX_SWEEPS = 16, EIG_MAX_REFINE = 6, EIG_ORTH_FROM = 4;   // the last two refinement steps only orthonormalise
constexpr float EIG_EXIT_COS2 = 1e-4f;                  // last FP32 sweep: its rotations and two refinement steps square this three times
constexpr float EIG_TIGHT_COS2 = 1e-11f;                // as orthogonal as FP32 columns get
__host__ __device__ constexpr size_t eig_smem(int n) {  // L, U, W, E in FP64, Y in FP32
  const int n8 = (n + 7) & ~7;
  return sizeof(double) * 4 * (size_t)n8 * (n8 + 4) + sizeof(float) * (size_t)n8 * n8;
}

__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// component-wise (plain FP32 instructions: the packed two-wide forms made a round of the Jacobi phase 10 % longer)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y)); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }
// Two independent rotations (x and y components): each makes two columns orthogonal, |y_p|^2 = a, |y_q|^2 = b, <y_p, y_q> = g;
// (p, q) <- (c p - s q, s p + c q).  a and b become the squared lengths after the rotation.
__device__ __forceinline__ void jacobi_rot2(float2& a, float2& b, float2 g, float exit_cos2, float2& c, float2& s, bool& above) {
  const float2 ab = mul2(a, b), gg = mul2(g, g);
  const bool on_x = gg.x > 1e-14f * ab.x, on_y = gg.y > 1e-14f * ab.y;
  above |= gg.x > exit_cos2 * ab.x;
  above |= gg.y > exit_cos2 * ab.y;
  g.x = on_x ? g.x : 0.0f; g.y = on_y ? g.y : 0.0f;
  // tan(theta) = 2g / (d + sign(d) sqrt(d^2 + 4g^2)), d = b - a: the smaller root.  With cos(2 theta) = |d| / hyp and
  // sin(2 theta) = +-2g / hyp:  cos^2 = (1 + cos 2theta) / 2, sin = sin(2 theta) / (2 cos): two reciprocal square roots.
  // (The 1e-37 keeps 0 / 0 out of the couple that needs no rotation; the norms are scaled to a largest value near one.)
  const float2 d = fma2(a, make_float2(-1.0f, -1.0f), b), g2 = add2(g, g), hd = mul2(d, make_float2(0.5f, 0.5f));
  const float2 h2 = fma2(g2, g2, fma2(d, d, make_float2(1e-37f, 1e-37f)));
  const float2 rh = make_float2(rsqrt_ftz(h2.x), rsqrt_ftz(h2.y));
  float2 cc = make_float2(fmaf(fabsf(hd.x), rh.x, 0.5f), fmaf(fabsf(hd.y), rh.y, 0.5f));
  cc.x = on_x ? cc.x : 1.0f; cc.y = on_y ? cc.y : 1.0f;
  const float2 rs = make_float2(rsqrt_ftz(cc.x), rsqrt_ftz(cc.y));
  const float2 sg = make_float2(__uint_as_float(__float_as_uint(g.x) ^ (__float_as_uint(d.x) & 0x80000000u)),
                                __uint_as_float(__float_as_uint(g.y) ^ (__float_as_uint(d.y) & 0x80000000u)));
  s = mul2(mul2(sg, rh), rs);
  c = mul2(cc, rs);
  const float2 tg = mul2(mul2(s, rs), g);   // tan(theta) g
  a = add2(a, neg2(tg));
  b = add2(b, tg);
}

// Makes the four columns of two blocks, a = (0, 1) and b = (2, 3), orthogonal between the blocks (and, with `within`, inside them
// first): LANES lanes hold R rows each.  n01, n23: squared lengths, carried along.  The rotations are worked out on the 4 x 4 Gram
// matrix: its six inner products are reduced together, and the second half round's follow from the first's by rotation.
template <int R, int LANES>
__device__ __forceinline__ void block_rotate(float2 (&a)[R], float2 (&b)[R], float2& n01, float2& n23, bool within, float exit_cos2, bool& above) {
  float g01 = 0.0f, g23 = 0.0f, g03 = 0.0f, g12 = 0.0f;
  float2 gx = make_float2(0.0f, 0.0f);                  // <0, 2>, <1, 3>
#pragma unroll
  for (int t = 0; t < R; ++t) {
    gx = fma2(a[t], b[t], gx);
    g03 = fmaf(a[t].x, b[t].y, g03); g12 = fmaf(a[t].y, b[t].x, g12);
    g01 = fmaf(a[t].x, a[t].y, g01); g23 = fmaf(b[t].x, b[t].y, g23);
  }
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) {
    gx.x += __shfl_xor_sync(0xFFFFFFFFu, gx.x, o); gx.y += __shfl_xor_sync(0xFFFFFFFFu, gx.y, o);
    g01 += __shfl_xor_sync(0xFFFFFFFFu, g01, o); g23 += __shfl_xor_sync(0xFFFFFFFFu, g23, o);
    g03 += __shfl_xor_sync(0xFFFFFFFFu, g03, o); g12 += __shfl_xor_sync(0xFFFFFFFFu, g12, o);
  }
  float2 c, s;
  if (within) {
    float2 na = make_float2(n01.x, n23.x), nb = make_float2(n01.y, n23.y);
    jacobi_rot2(na, nb, make_float2(g01, g23), exit_cos2, c, s, above);
    n01 = make_float2(na.x, nb.x); n23 = make_float2(na.y, nb.y);
    const float c02 = c.x * gx.x - s.x * g12, c03 = c.x * g03 - s.x * gx.y, c12 = s.x * gx.x + c.x * g12, c13 = s.x * g03 + c.x * gx.y;
    gx.x = c.y * c02 - s.y * c03; g03 = s.y * c02 + c.y * c03; g12 = c.y * c12 - s.y * c13; gx.y = s.y * c12 + c.y * c13;
    g01 = 0.0f; g23 = 0.0f;
#pragma unroll
    for (int t = 0; t < R; ++t) {
      a[t] = make_float2(c.x * a[t].x - s.x * a[t].y, s.x * a[t].x + c.x * a[t].y);
      b[t] = make_float2(c.y * b[t].x - s.y * b[t].y, s.y * b[t].x + c.y * b[t].y);
    }
  }
  jacobi_rot2(n01, n23, gx, exit_cos2, c, s, above);    // couples (0, 2) and (1, 3)
  const float x01 = c.x * g01 - s.x * g12, x03 = c.x * g03 - s.x * g23;        // <0', 1>, <0', 3>
  const float x21 = s.x * g01 + c.x * g12, x23 = s.x * g03 + c.x * g23;        // <2', 1>, <2', 3>
  const float2 gy = make_float2(s.y * x01 + c.y * x03, c.y * x21 - s.y * x23); // <0', 3'>, <1', 2'>
  float2 n32 = make_float2(n23.y, n23.x), c2, s2;
  jacobi_rot2(n01, n32, gy, exit_cos2, c2, s2, above);  // couples (0, 3) and (1, 2)
  n23 = make_float2(n32.y, n32.x);
  const float2 ns = neg2(s), ns2 = neg2(s2);
#pragma unroll
  for (int t = 0; t < R; ++t) {
    const float2 a1 = fma2(c, a[t], mul2(ns, b[t])), b1 = fma2(s, a[t], mul2(c, b[t]));
    const float2 bs = make_float2(b1.y, b1.x);
    a[t] = fma2(c2, a1, mul2(ns2, bs));
    const float2 b2 = fma2(s2, a1, mul2(c2, bs));
    b[t] = make_float2(b2.y, b2.x);
  }
}

template <int NT8>                                      // n rounded up to a multiple of eight, over eight
__global__ void __launch_bounds__(EIG_THREADS, 1)
eig_kernel(const double* __restrict__ gm, int n, int ld, double* __restrict__ evals, double* __restrict__ evecs) {
  metis_pdl_wait();
  constexpr int N8 = 8 * NT8, P = N8 + 4;
  constexpr int R = NT8, RP = N8;                       // rows per lane, rows of a column in Y
  constexpr int NB = N8 / 2;                            // column blocks of two (an even number)
  constexpr int GROUPS = NB / 2, JT = (8 * GROUPS + 31) / 32 * 32;             // groups of eight lanes, threads of the Jacobi phase
  extern __shared__ __align__(16) unsigned char esm[];
  double* Lm = reinterpret_cast<double*>(esm);
  double* U = Lm + N8 * P;
  double* W = U + N8 * P;
  double* E = W + N8 * P;
  float2* Yb = reinterpret_cast<float2*>(E + N8 * P);   // [block][RP rows] of (column 2b, column 2b + 1)
  __shared__ double lam[N8], inv_s[N8];
  __shared__ __align__(8) float nrm[N8];
  __shared__ int perm[N8], order[N8];
  __shared__ double gmax_s;
  __shared__ int flags[2][EIG_MAX_SWEEPS], flags64[EIG_MAX_SWEEPS];
  __shared__ unsigned int emax_s[2][EIG_MAX_REFINE];
  __shared__ float en_w[EIG_THREADS / 32];
  __shared__ uint8_t pairs[NB][GROUPS][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;

  // ---- sort by the diagonal, factorise ----
  for (int o = tid; o < N8 * N8; o += EIG_THREADS) {
    const int i = o / N8, j = o % N8;
    E[i * P + j] = (i < n && j < n) ? gm[i * ld + j] : (i == j ? -1.0 : 0.0);
  }
  if (tid < N8) perm[tid] = tid;
  if (tid < EIG_MAX_SWEEPS) flags[0][tid] = flags[1][tid] = flags64[tid] = 0;
  if (tid < EIG_MAX_REFINE) emax_s[0][tid] = emax_s[1][tid] = 0u;
  for (int o = tid; o < (NB - 1) * GROUPS; o += EIG_THREADS) {                  // round-robin tournament of the blocks
    const int step = o / GROUPS, m = o % GROUPS;
    const int a = m == 0 ? 0 : (step + m) % (NB - 1) + 1, b = m == 0 ? step % (NB - 1) + 1 : (step + NB - 1 - m) % (NB - 1) + 1;
    pairs[step][m][0] = (uint8_t)min(a, b); pairs[step][m][1] = (uint8_t)max(a, b);
  }
  __syncthreads();
  if (tid < 4 * N8) {                                   // rank of the diagonal entries, four lanes per entry
    const int e = tid >> 2;
    const double d = E[e * P + e];
    int rank = 0;
    for (int j = tid & 3; j < N8; j += 4) { const double x = E[j * P + j]; rank += (x > d) || (x == d && j < e); }
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 1);
    rank += __shfl_xor_sync(0xFFFFFFFFu, rank, 2);
    if ((tid & 3) == 0) {
      if (e < n) perm[rank] = e;                        // NaNs may collide; every entry stays a valid index
      if (rank == 0) gmax_s = d;
    }
  }
  __syncthreads();
  for (int o = tid; o < N8 * N8; o += EIG_THREADS) {
    const int i = o / N8, j = o % N8;
    Lm[i * P + j] = (i < n && j < n) ? 0.5 * (E[perm[i] * P + perm[j]] + E[perm[j] * P + perm[i]]) : 0.0;
  }
  const double gmax = gmax_s;
  __syncthreads();
  cta_cholesky<P>(Lm, n, 1e-14 * gmax, inv_s, nullptr, EIG_THREADS);
  // FP32 copy, scaled to a largest entry near one
  int ex = 0;
  if (gmax > 0.0 && gmax < 1e300) { (void)frexp(gmax, &ex); ex = (ex + 1) / 2; }
  const double y_scale = ldexp(1.0, -ex);
  for (int o = tid; o < NB * RP; o += EIG_THREADS) {
    const int b = o / RP, r = o % RP;
    float2 y = make_float2(0.0f, 0.0f);
    if (r < n) {
      if (r >= 2 * b) y.x = (float)(Lm[r * P + 2 * b] * y_scale);
      if (r >= 2 * b + 1) y.y = (float)(Lm[r * P + 2 * b + 1] * y_scale);
    }
    Yb[o] = y;
  }
  for (int o = tid; o < N8 * N8; o += EIG_THREADS) {   // the factor's upper triangle (the factorisation leaves the input there)
    const int i = o / N8, j = o % N8;
    if (j > i) Lm[i * P + j] = 0.0;
  }
  __syncthreads();

  double *X = U, *Wb = W;                               // the current vectors; the next ones overwrite W
  constexpr int N_WARPS = EIG_THREADS / 32, TRI = NT8 * (NT8 + 1) / 2, TPW = (TRI + N_WARPS - 1) / N_WARPS;
  int t_i[TPW], t_j[TPW];                               // this warp's lower tiles of S and R
#pragma unroll
  for (int u = 0; u < TPW; ++u) {
    const int o = warp + u * N_WARPS;
    int ti = 0;
    while ((ti + 1) * (ti + 2) / 2 <= o) ++ti;
    t_i[u] = ti; t_j[u] = o - ti * (ti + 1) / 2;
  }
  int still_open = 0;                                   // pairs left to the FP64 sweeps
  bool orth_only = false;
  for (int attempt = 0; attempt < 2; ++attempt) {
    const float exit_cos2 = attempt == 0 ? EIG_EXIT_COS2 : EIG_TIGHT_COS2;
    bool again = false;
    X = U; Wb = W;
    // ---- one-sided block Jacobi in FP32 on JT threads ----
    if (tid < JT) {
      auto bar = [] { asm volatile("bar.sync 1, %0;" ::"n"(JT) : "memory"); };
      const int m = tid >> 3, sub = tid & 7;
      const bool active = m < GROUPS;
      const int mc = min(m, GROUPS - 1);                // groups beyond the last one repeat its work and store nothing
      float2* nrm2 = reinterpret_cast<float2*>(nrm);
      // A group's access is 64 of a 128-byte line.  With an even number of chunks of eight rows, odd groups walk them in the
      // order 1, 0, 3, 2, ..., so that the two groups of a half warp never meet in the same banks (n = 64: a sixth off a
      // round); an odd number would need a padding chunk, which costs more than the conflicts.
      const int odd = R % 2 == 0 ? m & 1 : 0;
      auto row_of = [&](int t) { return sub + 8 * (t ^ odd); };
      for (int sweep = 0; sweep < EIG_MAX_SWEEPS; ++sweep) {
        // squared column norms: a group takes blocks 2m and 2m + 1
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float2 sq = make_float2(0.0f, 0.0f);
#pragma unroll
          for (int t = 0; t < R; ++t) { const float2 y = Yb[(2 * mc + h) * RP + sub + 8 * t]; sq = fma2(y, y, sq); }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) { sq.x += __shfl_xor_sync(0xFFFFFFFFu, sq.x, o); sq.y += __shfl_xor_sync(0xFFFFFFFFu, sq.y, o); }
          if (active && sub == 0) nrm2[2 * m + h] = sq;
        }
        int p = pairs[0][mc][0], r = pairs[0][mc][1];
        bar();
        bool above = false;
        for (int step = 0; step < NB - 1; ++step) {
          float2* yp = Yb + p * RP;
          float2* yr = Yb + r * RP;
          float2 a[R], b[R];                              // columns (0, 1) and (2, 3)
#pragma unroll
          for (int t = 0; t < R; ++t) { a[t] = yp[row_of(t)]; b[t] = yr[row_of(t)]; }
          const int pn = pairs[step + 1][mc][0], rn = pairs[step + 1][mc][1];  // (the table has a row more than it fills)
          float2 n01 = nrm2[p], n23 = nrm2[r];
          block_rotate<R, 8>(a, b, n01, n23, step == 0, exit_cos2, above);
          if (active) {
#pragma unroll
            for (int t = 0; t < R; ++t) { yp[row_of(t)] = a[t]; yr[row_of(t)] = b[t]; }
            if (sub == 0) { nrm2[p] = n01; nrm2[r] = n23; }
          }
          p = pn; r = rn;
          bar();
        }
        if (__any_sync(0xFFFFFFFFu, above && active) && lane == 0) flags[attempt][sweep] = 1;
        bar();
        if (!flags[attempt][sweep]) break;
      }
      // reciprocal column lengths in FP64 (0 for a zero column)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        double sx = 0.0, sy = 0.0;
#pragma unroll
        for (int t = 0; t < R; ++t) {
          const float2 y = Yb[(2 * mc + h) * RP + sub + 8 * t];
          sx = fma((double)y.x, (double)y.x, sx); sy = fma((double)y.y, (double)y.y, sy);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) { sx += __shfl_xor_sync(0xFFFFFFFFu, sx, o); sy += __shfl_xor_sync(0xFFFFFFFFu, sy, o); }
        if (active && sub < 2) {
          const double v = sub == 0 ? sx : sy;
          inv_s[2 * (2 * m + h) + sub] = v > 0.0 ? rsqrt64(v) : 0.0;
        }
      }
    }
    __syncthreads();

    // ---- U = normalised columns (zero columns stay zero) ----
    for (int o = tid; o < N8 * N8; o += EIG_THREADS) {
      const int i = o / N8, j = o % N8;
      U[i * P + j] = (double)(reinterpret_cast<const float*>(Yb + (j >> 1) * RP + i)[j & 1]) * inv_s[j];
    }
    __syncthreads();

    // ---- FP64 refinement ----
    for (int it = 0; it < EIG_MAX_REFINE; ++it) {
      for (int o = warp; o < NT8 * NT8; o += N_WARPS) {   // W = L^T X (L is lower triangular: k starts at the tile's own columns)
        const int ti = o / NT8, tj = o % NT8;
        double acc[2] = {0.0, 0.0}, acc2[2] = {0.0, 0.0};
#pragma unroll
        for (int t = 0; t < NT8; ++t) {
          if (t < ti) continue;
          const int kk = 8 * t + q;
          dmma(acc, Lm[kk * P + 8 * ti + g], X[kk * P + 8 * tj + g]);
          dmma(acc2, Lm[(kk + 4) * P + 8 * ti + g], X[(kk + 4) * P + 8 * tj + g]);
        }
        Wb[(8 * ti + g) * P + 8 * tj + 2 * q] = acc[0] + acc2[0];
        Wb[(8 * ti + g) * P + 8 * tj + 2 * q + 1] = acc[1] + acc2[1];
      }
      __syncthreads();
      double sv[TPW][2], rv[TPW][2];                      // lower tiles of S and of X^T X
#pragma unroll
      for (int u = 0; u < TPW; ++u) {
        sv[u][0] = sv[u][1] = rv[u][0] = rv[u][1] = 0.0;
        const int o = warp + u * N_WARPS;
        if (o < TRI) {
          const int ti = t_i[u], tj = t_j[u];
#pragma unroll
          for (int kk = 0; kk < N8; kk += 4) {
            dmma(sv[u], Wb[(kk + q) * P + 8 * ti + g], Wb[(kk + q) * P + 8 * tj + g]);
            dmma(rv[u], X[(kk + q) * P + 8 * ti + g], X[(kk + q) * P + 8 * tj + g]);
          }
          if (ti == tj && (g >> 1) == q) {                // lane holds the diagonal entry 8 ti + g
            const double ss = (g & 1) ? sv[u][1] : sv[u][0], rr = (g & 1) ? rv[u][1] : rv[u][0];
            lam[8 * ti + g] = rr > 0.0 ? ss / rr : 0.0;
            inv_s[8 * ti + g] = rr;                       // squared length: zero for a zero column
          }
        }
      }
      __syncthreads();
      orth_only |= it >= EIG_ORTH_FROM;
      bool open = false;
      float em = 0.0f, en = 0.0f;
#pragma unroll
      for (int u = 0; u < TPW; ++u) {
        const int o = warp + u * N_WARPS;
        if (o < TRI) {
          const int ti = t_i[u], tj = t_j[u];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int i = 8 * ti + g, j = 8 * tj + 2 * q + e;
            const double r = (i == j ? 1.0 : 0.0) - rv[u][e];
            double e_ij = 0.5 * r, e_ji = 0.5 * r;
            if (i != j) {
              if (inv_s[i] == 0.0 || inv_s[j] == 0.0) { e_ij = 0.0; e_ji = 0.0; }
              else if (!orth_only) {
                const double gap = lam[j] - lam[i], a = sv[u][e] + lam[j] * r, b = sv[u][e] + lam[i] * r;
                if (sv[u][e] * sv[u][e] > 1e-28 * fabs(lam[i] * lam[j])) {         // orthogonal to FP64 rounding: nothing to rotate
                  if (fabs(a) < 0.0625 * fabs(gap) && fabs(b) < 0.0625 * fabs(gap)) {
                    const double rg = 1.0 / gap;
                    e_ij = a * rg; e_ji = -b * rg;
                  } else if (sv[u][e] * sv[u][e] > 1e-24 * fabs(lam[i] * lam[j])) open = true;
                }
              }
            } else if (inv_s[i] == 0.0) e_ij = e_ji = 0.0;
            em = fmaxf(em, fmaxf(fabsf((float)e_ij), fabsf((float)e_ji)));
            en = fmaf((float)e_ij, (float)e_ij, fmaf((float)e_ji, (float)e_ji, en));
            E[i * P + j] = e_ij;
            if (ti != tj) E[j * P + i] = e_ji;            // a diagonal tile computes both of its triangles
          }
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) { em = fmaxf(em, __shfl_xor_sync(0xFFFFFFFFu, em, o)); en += __shfl_xor_sync(0xFFFFFFFFu, en, o); }
      if (lane == 0) { atomicMax(&emax_s[attempt][it], __float_as_uint(em)); en_w[warp] = en; }
      still_open = __syncthreads_or(open ? 1 : 0);
      float norm2 = 0.0f;                                 // squared norm of E (diagonal-tile pairs twice), the same sum in every thread
#pragma unroll
      for (int w = 0; w < N_WARPS; ++w) norm2 += en_w[w];
      if (still_open || !(norm2 < 0.0625f)) {
        if (attempt == 0) { again = true; break; }        // back to the FP32 sweeps, with the tight exit test
        still_open = 1;
        if (!(norm2 < 0.0625f)) { orth_only = true; continue; }                    // the same step once more, pairs only orthonormalised
      }
      for (int o = warp; o < NT8 * NT8; o += N_WARPS) {   // X E + X into the buffer of W
        const int ti = o / NT8, tj = o % NT8;
        double acc[2] = {0.0, 0.0}, acc2[2] = {0.0, 0.0};
#pragma unroll
        for (int kk = 0; kk < N8; kk += 8) {
          dmma(acc, X[(8 * ti + g) * P + kk + q], E[(kk + q) * P + 8 * tj + g]);
          dmma(acc2, X[(8 * ti + g) * P + kk + 4 + q], E[(kk + 4 + q) * P + 8 * tj + g]);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int at = (8 * ti + g) * P + 8 * tj + 2 * q + e;
          Wb[at] = X[at] + (acc[e] + acc2[e]);
        }
      }
      __syncthreads();
      double* tmp = X; X = Wb; Wb = tmp;
      if (__uint_as_float(emax_s[attempt][it]) < 2e-7f) break;     // the next correction would be this one squared (a NaN runs all steps)
    }

    if (!again) break;
    __syncthreads();
  }
  __syncthreads();
  // ---- pairs the refinement could not separate: FP64 one-sided Jacobi on the columns of W = L^T X ----
  if (still_open || orth_only) {
    for (int o = tid; o < N8 * N8; o += EIG_THREADS) {
      const int i = o / N8, j = o % N8;
      double a = 0.0;
      for (int k = i; k < N8; ++k) a = fma(Lm[k * P + i], X[k * P + j], a);
      Wb[i * P + j] = a;
    }
    __syncthreads();
    const int m = tid >> 3, sub = tid & 7;
    const bool active = m < N8 / 2;
    for (int sweep = 0; sweep < EIG_MAX_SWEEPS; ++sweep) {
      bool above = false;
      for (int step = 0; step < N8 - 1; ++step) {       // round-robin tournament of the columns
        const int mm = active ? m : 0;
        const int p = mm == 0 ? 0 : (step + mm) % (N8 - 1) + 1, r = mm == 0 ? step % (N8 - 1) + 1 : (step + N8 - 1 - mm) % (N8 - 1) + 1;
        double a = 0.0, b = 0.0, c = 0.0;
#pragma unroll
        for (int t = 0; t < NT8; ++t) {
          const double x = Wb[(sub + 8 * t) * P + p], y = Wb[(sub + 8 * t) * P + r];
          a = fma(x, x, a); b = fma(y, y, b); c = fma(x, y, c);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          a += __shfl_xor_sync(0xFFFFFFFFu, a, o); b += __shfl_xor_sync(0xFFFFFFFFu, b, o); c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
        }
        __syncwarp();
        if (active && c * c > 1e-30 * (a * b)) {
          above |= c * c > 1e-13 * (a * b);
          const double d = b - a, rh = rsqrt64(fma(4.0 * c, c, d * d));
          const double cc = fma(0.5 * fabs(d), rh, 0.5), rs = rsqrt64(cc);
          const double cs = cc * rs, sn = (d < 0.0 ? -c : c) * rh * rs;
#pragma unroll
          for (int t = 0; t < NT8; ++t) {
            const int row = (sub + 8 * t) * P;
            const double x = Wb[row + p], y = Wb[row + r], u = X[row + p], v = X[row + r];
            Wb[row + p] = cs * x - sn * y; Wb[row + r] = sn * x + cs * y;
            X[row + p] = cs * u - sn * v; X[row + r] = sn * u + cs * v;
          }
        }
        __syncthreads();
      }
      if (above) flags64[sweep] = 1;
      __syncthreads();
      if (!flags64[sweep]) break;
    }
    if (tid < N8) {
      double a = 0.0;
      for (int i = 0; i < N8; ++i) a = fma(Wb[i * P + tid], Wb[i * P + tid], a);
      lam[tid] = a;
    }
    __syncthreads();
  }

  // ---- eigenvalues descending, eigenvectors in the input's row order ----
  if (tid < n) order[tid] = tid;                        // stays a valid index if NaNs make the ranks below collide
  __syncthreads();
  if (tid < n) {
    const double li = lam[tid];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += (lam[j] > li) || (lam[j] == li && j < tid);
    order[rank] = tid;
  }
  __syncthreads();
  if (tid < n) evals[tid] = lam[order[tid]] + 0.0 * gmax;                      // a non-finite matrix is seen by the status check
  for (int o = tid; o < n * n; o += EIG_THREADS) {
    const int i = o / n, j = o % n;
    evecs[perm[i] * n + j] = X[i * P + order[j]];
  }
}

}  // namespace metis_small
