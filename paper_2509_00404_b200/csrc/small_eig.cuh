// One-CTA dense linear algebra of a decomposition (n <= 72): FP64 Cholesky factorisation and the symmetric
// eigen-decomposition.  Both are latency chains on one SM, so what counts is the number of dependent steps and how long one is.
#pragma once
#include <type_traits>

#include "common.cuh"
#include "reciprocal.cuh"
#include "tridiag.cuh"

namespace metis_small {

constexpr int MAXQ = 72;                                // k + p at most (k = 64 with p = 8)
constexpr int PITCH = MAXQ + 4;                         // doubles; 4 or 12 mod 16: every fragment access below is conflict-free

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

// In-place Cholesky factorisation of the lower triangle of Y (n x n, n8 = n rounded up to a multiple of eight, row pitch P doubles (even),
// rows and columns up to n8 must exist and be zero beyond n), called by all nthr threads (at least two warps and n8 - 8 threads).
// Panels of eight columns: every thread factorises the panel's diagonal block for itself in registers (a column is a reciprocal root and two operations
// deep, without an exchange: with a row of the block per lane it was a broadcast of the pivot deeper and 36 double shuffles a panel, 2200 cycles with the
// trailing update against 1500) and carries one row below it along; then all warps but the last, which stores the block, subtract the panel's rank-8 product from the trailing tiles
// on the FP64 tensor cores, two tiles at a time.  (One barrier per column with the matrix spread over 256 threads' registers took 800 cycles a
// column.)  A pivot not above `tol` marks a dependent column: it takes no part in the updates and ends as a zero column with
// inv_out[j] = 0; otherwise inv_out[j] = 1 / L[j][j].  *dmin_out (optional): the smallest accepted pivot, to 20 bits from below.  tid, bar: index within the group of nthr
// threads and the group's barrier.
template <int P, class Bar>
__device__ __forceinline__ void group_cholesky(double* Y, int n, double tol, double* inv_out, double* dmin_out, int tid, int nthr, Bar bar) {
  const int lane = tid & 31, warp = tid >> 5, n_warps = nthr >> 5;
  const int n8 = (n + 7) & ~7, g = lane >> 2, q = lane & 3;
  int dmin = 0x7FE00000;                                // of the smallest accepted pivot, its high word
  for (int c0 = 0; c0 < n8; c0 += 8) {
    const int r = c0 + 8 + 32 * warp + lane;            // a row below the block
    const bool busy = warp == n_warps - 1 || c0 + 8 + 32 * warp < n8;
    double a[8][8], inv[8];                             // the block's lower triangle
    if (busy) {
      double v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int c = 0; c <= i; c += 2) {
          const double2 x = *reinterpret_cast<const double2*>(Y + (c0 + i) * P + c0 + c);
          a[i][c] = x.x;
          if (c < i) a[i][c + 1] = x.y;
        }
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = r < n8 ? Y[r * P + c0 + c] : 0.0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const double d = a[j][j], rs = rsqrt_cubic(d);  // (selected, not branched around)
        const bool on = d > tol;
        inv[j] = on ? rs : 0.0;
        dmin = min(dmin, on ? __double2hiint(d) : 0x7FE00000);
#pragma unroll
        for (int i = j; i < 8; ++i) a[i][j] *= inv[j];
        v[j] *= inv[j];
#pragma unroll
        for (int c = j + 1; c < 8; ++c) {
#pragma unroll
          for (int i = c; i < 8; ++i) a[i][c] = fma(-a[i][j], a[c][j], a[i][c]);
          v[c] = fma(-v[j], a[c][j], v[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < 8; ++c) if (r < n8) Y[r * P + c0 + c] = v[c];
    }
    bar();                                    // the block has been read by every warp: its factor may be stored
    if (warp == n_warps - 1) {                          // while the others go on; every lane stores all of it (a row per lane: a branch of 200 cycles for each)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (c0 + i < n) inv_out[c0 + i] = inv[i];
#pragma unroll
        for (int c = 0; c < 8; c += 2)
          *reinterpret_cast<double2*>(Y + (c0 + i) * P + c0 + c) = make_double2(c <= i ? a[i][c] : 0.0, c < i ? a[i][c + 1] : 0.0);
      }
    }
    // trailing tiles (ti >= tj > panel): Y -= L_panel L_panel^T
    const int first = c0 / 8 + 1, nt = n8 / 8 - first, tiles = nt * (nt + 1) / 2;
    for (int o = warp; o < tiles && warp < n_warps - 1; o += 2 * (n_warps - 1)) {
      double acc[2][2], a[2][2], b[2][2];
      double* out[2];
      const bool two = o + n_warps - 1 < tiles;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        int ti, tj;
        lower_tile(u == 0 || !two ? o : o + n_warps - 1, ti, tj);
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
    bar();
  }
  if (dmin_out != nullptr && tid == nthr - 1) *dmin_out = __hiloint2double(dmin, 0);
  bar();
}

template <int P>
__device__ __forceinline__ void cta_cholesky(double* Y, int n, double tol, double* inv_out, double* dmin_out, int nthr) {
  group_cholesky<P>(Y, n, tol, inv_out, dmin_out, (int)threadIdx.x, nthr, [] { __syncthreads(); });
}

// The inverse of diagonal block b of the factor of cta_cholesky (8 x 8, into X with row pitch xp), by one warp (lane = column).  inv: reciprocal
// pivots (zero for a dependent column, whose row of the inverse is then zero).
template <int P>
__device__ __forceinline__ void invert_diagonal_block(const double* L, const double* inv, int n, int b, double* X, int xp) {
  const int lane = threadIdx.x & 31;
  if (lane < 8) {
    double x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      double s = 0.0;
#pragma unroll
      for (int k = 0; k < i; ++k) s = fma(L[(8 * b + i) * P + 8 * b + k], x[k], s);
      const double r = 8 * b + i < n ? inv[8 * b + i] : 0.0;
      x[i] = i == lane ? r : (i > lane ? -r * s : 0.0);
      X[i * xp + lane] = x[i];
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Symmetric positive semi-definite eigen-decomposition in one CTA.
//   1. Householder reduction to a tridiagonal matrix T in FP64 (tridiag.cuh), the matrix in the registers of four threads per row.
//      A step is a chain through one more warp, which works out the scalars, the vectors of the update and the next column: product, its sum with x,
//      the update, the next product, 640 cycles at n = 40 (FP64 operation 8, matrix instruction 26, 64-bit shuffle with addition 35, shared-memory
//      round trip 29, barrier 20 to 40).  What counts is how long the two chains are - the other warps' from the vectors to the next product and the
//      scalars' warp's through the next reflector - and the bytes that the vectors bring into registers (128 a cycle: at n = 72 half of a step).
//      Every thread working out the scalars for itself made it 1000 cycles, three barriers with the column published by its owner 1050.
//      Meanwhile six warps sort the matrix by descending diagonal and factorise it, G = L L^T (dependent columns zeroed);
//   2. eigenvalues of T by multisection on Sturm counts to a relative 2^-30 of themselves, eigenvectors by twisted factorisations
//      (Dhillon and Parlett, "Orthogonal eigenvectors and relative gaps", 2003, without their representation tree), taken back through
//      the reflectors in panels of eight (compact WY) on the FP64 tensor cores;
//   3. FP64 refinement of the eigenvectors U (Ogita and Aishima, "Iterative refinement for symmetric eigenvalue
//      decomposition", 2018): with R = I - U^T U and S = U^T G U, U += U E, E_ij = (S_ij + s_j R_ij) / (s_j - s_i), E_ii = R_ii / 2,
//      s_i = S_ii / (1 - R_ii); the error is squared by each step.  S is formed as W^T W with W = L^T U, which keeps the
//      relative accuracy of small eigenvalues, of which T keeps only the absolute one.  The products run on the FP64 tensor cores.
//      One step is enough unless eigenvalues lie closer than a hundredth of a per cent or so;
//   4. eigenvalues that agree to about 1e-9 come out of step 2 with dependent vectors (|E_ij| above 1/16, or E as a whole not
//      small): then one-sided Jacobi on the columns of L in FP32 makes the start instead (Y = L J with orthogonal columns; eight lanes
//      own two blocks of two columns: one round loads four columns, forms their six inner products at once, works out the
//      four rotations between the blocks on the 4 x 4 Gram matrix in registers and applies them, 784 cycles at n = 40) and
//      step 3 is repeated; if pairs are still open after that, they are only orthonormalised in step 3 and FP64
//      one-sided Jacobi sweeps on the columns of W = L^T U, U rotated along, finish the work (repeated eigenvalues).
// Precision, n = 8 ... 72, in 80 bits (in brackets: with the FP32 sweeps as every start): U^T G U diagonal to 2e-15 (2e-12) of its largest
// entry, and to 1e-14, 1e-13 and 4e-12 (4e-12, 3e-11 and 9e-10) of sqrt(lambda_i lambda_j) where the eigenvalues span two, four and six decades (the factor's
// rounding), U orthonormal to 1e-15 (1e-13); eigenvalues within 4e-5 of each other 3e-14 and 1e-13 (6e-8 and 1e-14); half of them repeated
// 1e-8 and 3e-9 (7e-8 and 2e-8).  A pair of W that is orthogonal already is left to the orthonormalisation alone, half of R_ij to either column, only
// if that does not tilt it: between eigenvalues of different size it does, by half of R_ij times the root of their ratio.
// Input: `parts` partials of the Gram matrix (ld x ld each, leading n x n block used).  Output: eigenvalues descending, eigenvectors as columns of
// evecs[n][n].
// Measured alone, planted spectrum (in brackets: the reduction with three barriers a step, and the Jacobi sweeps of step 4 as the start of every
// matrix): n = 8 10.3 us (10.3, 12.5), n = 32 25.8 (32.8, 43), n = 40 34.9 (43.1, 64), n = 64 68 (88, 127), n = 72 93 (115, 242).  Nearly diagonal
// matrices are the ones the sweeps alone finish sooner (off the diagonal 1e-4 of it n = 32 21, n = 40 29, n = 72 80), and repeated eigenvalues pay for both starts.
// Cycles at n = 40: load 2.5 k, reduction 25 k, multisection 13 k + 2 k, vectors 5.6 k + 4.9 k, refinement 7.4 k, output 2.3 k.
// Four threads per row reduce the matrix while six warps factorise it; the products and the multisection use all of them.
constexpr int EIG_CHOL_THREADS = 192;
__host__ __device__ constexpr int eig_threads(int nt8) { return nt8 <= 1 ? 256 : 512; }
constexpr int EIG_MAX_SWEEPS = 16, EIG_MAX_REFINE = 6, EIG_ORTH_FROM = 4;   // the last two refinement steps only orthonormalise
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
__global__ void __launch_bounds__(eig_threads(NT8), 1)
eig_kernel(const double* __restrict__ gm, int parts, int n, int ld, double* __restrict__ evals, double* __restrict__ evecs) {
  metis_pdl_wait();
  constexpr int N8 = 8 * NT8, P = N8 + 4, EIG_THREADS = eig_threads(NT8);
  constexpr int TD = 4 * N8, TS = TD + 32;              // threads of the reduction: four per row, and the warp that works out its scalars
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
  __shared__ int flags[EIG_MAX_SWEEPS], flags64[EIG_MAX_SWEEPS];
  __shared__ __align__(16) double2 te[N8 + 8];          // diagonal and squared subdiagonal of the tridiagonal matrix (a block beyond it is read ahead)
  __shared__ __align__(16) double ys[N8], rs[2][N8], us[N8], ps[2][N8], qs[N8];
  __shared__ double eo[N8 + 1], beta_s[N8], v1_s[N8];
  __shared__ int pos[N8];
  __shared__ unsigned char grid_count[EIG_THREADS / 2];
  __shared__ __align__(16) double Tp[64 * NT8];
  __shared__ unsigned int emax_s[2][EIG_MAX_REFINE];
  __shared__ float en_w[EIG_THREADS / 32];
  __shared__ uint8_t pairs[NB][GROUPS][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;

  // ---- the matrix ----
  for (int o = tid; o < N8 * N8; o += EIG_THREADS) {
    const int i = o / N8, j = o % N8;
    double a = i == j ? -1.0 : 0.0;
    if (i < n && j < n) {
      const double* src = gm + i * ld + j;
      a = src[0];
      for (int p = 1; p < parts; p += 8) {              // the other partials, in their order, loads in flight
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = p + u < parts ? src[(p + u) * ld * ld] : 0.0;
#pragma unroll
        for (int u = 0; u < 8; ++u) a += v[u];
      }
    }
    E[i * P + j] = a;
  }
  if (tid < N8) perm[tid] = tid;
  if (tid < EIG_MAX_SWEEPS) flags[tid] = flags64[tid] = 0;
  if (tid < EIG_MAX_REFINE) emax_s[0][tid] = emax_s[1][tid] = 0u;
  __syncthreads();
  // an even power of two brings the largest entry near one; its root does for the FP32 copy of the factor
  int top = 0;
  for (int i = lane; i < n; i += 32) top = max(top, __double2hiint(E[i * P + i]));
  top = __reduce_max_sync(0xFFFFFFFFu, top) >> 20;
  const int ex = top > 0 && top < 2046 ? (top - 1022 + 1) >> 1 : 0;
  const double y_scale = __hiloint2double((1023 - ex) << 20, 0);
  double* V = W;                                        // row j: column j of the trailing matrix when it is reduced (reflector j)
  auto arrive = [](int id) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(TS) : "memory"); };
  auto await = [](int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(TS) : "memory"); };
  constexpr int Y_READY = 2, U_READY = 4, X_READY = 5;
  if (tid < TD) {
    // ---- Householder reduction: eight lanes hold rows i0 and i0 + 1 in registers (columns s8, s8 + 8, ...) ----
    const int s8 = tid & 7, i0 = 2 * (tid >> 3), last_row = (tid | 31) >> 2 | 1;
    double row[2][NT8], x[NT8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int t = 0; t < NT8; ++t) {
        const int c = s8 + 8 * t, i = i0 + h;
        row[h][t] = i < n && c < n ? 0.5 * (E[i * P + c] + E[c * P + i]) * (y_scale * y_scale) : 0.0;
      }
    if (tid < 8) {                                      // column 0; row 1
      if (tid == 0) te[0].x = row[0][0];
#pragma unroll
      for (int t = 0; t < NT8; ++t) { V[s8 + 8 * t] = s8 + 8 * t > 0 ? row[0][t] : 0.0; rs[0][s8 + 8 * t] = row[1][t]; }
    }
    await(X_READY);
#pragma unroll
    for (int t = 0; t < NT8; ++t) x[t] = V[s8 + 8 * t];
    // steps `from` ... `to` - 1, columns from 8 T0 on (those before are done)
    auto steps = [&](auto t0, int from, int to) {
      constexpr int T0 = decltype(t0)::value;
#pragma unroll 1
      for (int j = from; j < to; ++j) {
        const bool live = last_row > j;                   // the warp has a row below j
        if (live) {
          // the sums of eight lanes are those of two columns of a matrix product that each lane q, q + 4, ... gets, for rows 2 q and 2 q + 1
          // of the warp's eight: two matrix instructions and an addition (50 cycles; by shuffles 105)
          double y0 = 0.0, y1 = 0.0, d0[2] = {0.0, 0.0}, d1[2] = {0.0, 0.0};
#pragma unroll
          for (int t = T0; t < NT8; ++t) { y0 = fma(row[0][t], x[t], y0); y1 = fma(row[1][t], x[t], y1); }
          dmma(d0, 1.0, y0);
          dmma(d1, 1.0, y1);
          if (lane < 4) *reinterpret_cast<double2*>(ys + 8 * warp + 2 * lane) = make_double2(d0[0] + d0[1], d1[0] + d1[1]);
        }
        arrive(Y_READY);
        await(U_READY);
        if (live) {
          const double2 c = *reinterpret_cast<const double2*>(ps[j & 1] + i0);
#pragma unroll
          for (int t = T0; t < NT8; ++t) {
            const double u = us[s8 + 8 * t];
            row[0][t] = fma(c.x, u, row[0][t]);
            row[1][t] = fma(c.y, u, row[1][t]);
          }
        }
        await(X_READY);
        if (live) {
          const double2 c = *reinterpret_cast<const double2*>(qs + i0);
#pragma unroll
          for (int t = T0; t < NT8; ++t) {
            row[0][t] = fma(c.x, x[t], row[0][t]);
            row[1][t] = fma(c.y, x[t], row[1][t]);
            x[t] = V[(j + 1) * P + s8 + 8 * t];
          }
          double* out = rs[(j + 1) & 1] + s8;             // row j + 2 for the next step
          const bool even = i0 == j + 2, odd = i0 + 1 == j + 2;
#pragma unroll
          for (int t = T0; t < NT8; ++t) {
            if (even) out[8 * t] = row[0][t];
            if (odd) out[8 * t] = row[1][t];
          }
        }
      }
    };
    constexpr int SEG = NT8 >= 7 ? 3 : (NT8 >= 4 ? (NT8 + 1) / 2 : NT8);         // blocks of eight columns to a loop
    steps(std::integral_constant<int, 0>{}, 0, min(8 * SEG, n - 2));
    if (SEG < NT8) steps(std::integral_constant<int, SEG < NT8 ? SEG : 0>{}, 8 * SEG, min(16 * SEG, n - 2));
    if (2 * SEG < NT8) steps(std::integral_constant<int, 2 * SEG < NT8 ? 2 * SEG : 0>{}, 16 * SEG, n - 2);
#pragma unroll
    for (int h = 0; h < 2; ++h)                         // what is left of the last two rows
#pragma unroll
      for (int t = 0; t < NT8; ++t)
        if (s8 + 8 * t == n - 1) {
          if (i0 + h == n - 2) eo[n - 2] = row[h][t];
          if (i0 + h == n - 1) te[n - 1].x = row[h][t];
        }
  } else if (tid < TS) {
    // ---- the warp of the scalars, entries lane, lane + 32, ... of the vectors: with y = A x and r = A e_1 it is
    // A v = u = y - alpha r,  v^T A v = x^T y - 2 alpha y_1 + alpha^2 r_1;  w = beta u - K v,  A -= v w^T + w v^T = p u^T + q v^T.
    // p and u, which do not depend on K, go ahead of q; the next column it updates by itself, so that the others go from the update
    // to the next product without a barrier, and works out that column's reflector meanwhile.  Column j + 1 is not read again
    // except for its first entry, so x stands for v in the others' last term.
    // What orders the vectors (this warp only arrives at U_READY and X_READY, so the others may be a step behind): ys and rs of a step are written
    // behind its predecessor's X_READY and read behind its Y_READY; us and qs are written behind Y_READY, which the others reach when they have
    // read those of the step before; p goes out ahead of Y_READY, while they may still read the step before's, so it has two halves, like rs ----
    constexpr int OWN = (N8 + 31) / 32;
    // the sum of a warp, in each lane: sums of four lanes first as columns (each lane gets two of the eight), then as rows
    auto sum32 = [](double v) {
      double d[2] = {0.0, 0.0}, f[2] = {0.0, 0.0};
      dmma(d, 1.0, v);
      dmma(f, d[0] + d[1], 1.0);
      return f[0];
    };
    double x[OWN];
    await(X_READY);
#pragma unroll
    for (int k = 0; k < OWN; ++k) x[k] = lane + 32 * k < N8 ? V[lane + 32 * k] : 0.0;
    double x0 = V[1];
#pragma unroll 1
    for (int j = 0; j + 2 < n; ++j) {
      const double *rj = rs[j & 1], xb = V[j * P + j + 2];
      double sq = 0.0, xy = 0.0, y[OWN], v[OWN], r[OWN], alpha, beta;
#pragma unroll
      for (int k = 0; k < OWN; ++k) sq = fma(x[k], x[k], sq);
      metis_tri::reflector(x0, sum32(sq), alpha, beta);
      const double v1 = x0 - alpha, pa = -beta * v1;
#pragma unroll
      for (int k = 0; k < OWN; ++k) {
        const int e = lane + 32 * k;
        v[k] = e == j + 1 ? v1 : x[k];
        if (e < N8) ps[j & 1][e] = -beta * v[k];
      }
      eo[j] = alpha; beta_s[j] = beta; v1_s[j] = v1;
      await(Y_READY);                                   // the product and row j + 1 are there
#pragma unroll
      for (int k = 0; k < OWN; ++k) {
        const int e = min(lane + 32 * k, N8 - 1);
        y[k] = ys[e]; r[k] = rj[e];
      }
      const double ya = ys[j + 1], ra = rj[j + 1], yb = ys[j + 2], rb = rj[j + 2];
#pragma unroll
      for (int k = 0; k < OWN; ++k) {
        const int e = lane + 32 * k;
        xy = fma(x[k], y[k], xy);
        y[k] = e > j ? fma(-alpha, r[k], y[k]) : 0.0;   // now u
        if (e < N8) us[e] = y[k];
      }
      arrive(U_READY);
      xy = sum32(xy);
      const double ua = fma(-alpha, ra, ya), ba = -beta * ua, b2 = beta * beta, k0 = b2 * (alpha * fma(alpha, ra, -2.0 * ya));
      double xv[OWN];
#pragma unroll
      for (int k = 0; k < OWN; ++k) {                   // all of the next column but the term with K
        const int e = lane + 32 * k;
        const bool in = e > j + 1 && e < N8;
        r[k] = in ? fma(pa, y[k], fma(ba, v[k], r[k])) : 0.0;
        xv[k] = in ? v1 * v[k] : 0.0;
        y[k] *= -beta;
      }
      const double x0a = fma(pa, fma(-alpha, rb, yb), fma(ba, xb, rb)), x0b = v1 * xb;
      const double K2 = fma(b2, xy, k0);
#pragma unroll
      for (int k = 0; k < OWN; ++k) {
        const int e = lane + 32 * k;
        x[k] = fma(K2, xv[k], r[k]);
        if (e < N8) { qs[e] = fma(K2, v[k], y[k]); V[(j + 1) * P + e] = x[k]; }
      }
      arrive(X_READY);
      x0 = fma(K2, x0b, x0a);
      te[j + 1].x = fma(pa, ua, fma(fma(K2, v1, ba), v1, ra));
      __syncwarp();
    }
  } else if (tid < TS + EIG_CHOL_THREADS) {
    // ---- meanwhile: sorted by the diagonal and factorised ----
    auto bar = [] { asm volatile("bar.sync 3, %0;" ::"n"(EIG_CHOL_THREADS) : "memory"); };
    const int ct = tid - TS;
    for (int e = ct; e < N8; e += EIG_CHOL_THREADS) {
      const double d = E[e * P + e];
      int rank = 0;
#pragma unroll 8
      for (int j = 0; j < N8; ++j) { const double x = E[j * P + j]; rank += (x > d) || (x == d && j < e); }
      pos[e] = rank;
      if (e < n) perm[rank] = e;                        // NaNs may collide; every entry stays a valid index
      if (rank == 0) gmax_s = d;
    }
    bar();
    for (int o = ct; o < N8 * N8; o += EIG_CHOL_THREADS) {
      const int i = o / N8, j = o % N8;
      Lm[i * P + j] = (i < n && j < n) ? 0.5 * (E[perm[i] * P + perm[j]] + E[perm[j] * P + perm[i]]) : 0.0;
    }
    bar();
    group_cholesky<P>(Lm, n, 1e-14 * gmax_s, inv_s, nullptr, ct, EIG_CHOL_THREADS, bar);
  }
  __syncthreads();
  const double gmax = gmax_s;
  if (tid <= N8) {
    te[tid].y = tid > 0 && tid < n ? fmax(eo[tid - 1] * eo[tid - 1], metis_tri::TINY_SQUARE) : 0.0;
    if (tid >= n) te[tid].x = 4.0 * N8;
  }
  if (tid + 2 < n) V[tid * P + tid + 1] = v1_s[tid];
  for (int o = tid; o < N8 * N8; o += EIG_THREADS) {   // the factor's upper triangle (the factorisation leaves the input there)
    const int i = o / N8, j = o % N8;
    if (j > i) Lm[i * P + j] = 0.0;
  }
  const int rank = __syncthreads_count(tid < n && inv_s[tid < n ? tid : 0] > 0.0);
  // ---- eigenvalues and eigenvectors of the tridiagonal matrix, descending ----
  constexpr int GRID = EIG_THREADS / 2;                  // points that bring every eigenvalue to about a sixth of an octave
  const long long grid_lo = __double_as_longlong(0x1p-56), grid_w = (__double_as_longlong(2.0 * N8) - grid_lo) / GRID + 1;
  if (tid < GRID) {
    const double x[1] = {__longlong_as_double(grid_lo + grid_w * (tid + 1))};
    int c[1];
    metis_tri::sturm_counts<1>(te, NT8, x, c);
    grid_count[tid] = (unsigned char)c[0];
  }
  __syncthreads();
  double *Dp = E, *Z = U;                               // column e of each: vector e
  constexpr int TV = 4 * N8;                            // four threads per vector
  // Lanes per eigenvalue in the multisection, two points each, so that a warp (or two) runs on each of the four schedulers: a round at n = 40 is 1290
  // cycles, 1180 of them the Sturm sequences (three points on fewer warps: 1650).
  constexpr int LE = N8 <= 32 ? 4 : (N8 <= 40 || N8 > 64 ? 3 : 2), PW = 32 / LE, TE = (N8 + PW - 1) / PW * 32;
  {
    if (tid < TE) {
      const int e = PW * warp + min(lane / LE, PW - 1), below = max(n - 1 - e, 0);
      int at = 0;                                       // the first point with more than `below` eigenvalues under it
#pragma unroll
      for (int step = GRID / 2; step > 0; step >>= 1) if (grid_count[at + step - 1] <= below) at += step;
      const double v = metis_tri::multisect<LE, 2>(te, NT8, grid_lo + grid_w * at, grid_lo + grid_w * (at + 1), below,
                                                   LE == 4 ? 9 : (LE == 3 ? 10 : 12));
      if (lane % LE == 0 && lane / LE < PW && e < N8) lam[e] = v;
    }
  }
  __syncthreads();
  if (tid < TV) {
    auto bar = [] { asm volatile("bar.sync 2, %0;" ::"n"(TV) : "memory"); };
    if (tid < 2 * n) {                                  // pivots from the top and from the bottom
      const int e = tid >> 1, down = tid & 1;
      const double lm = lam[e];
      double* D = (down ? Z : Dp) + e;
      double pm = 0.0, p = 1.0;
#pragma unroll 1
      for (int b = 0; b < NT8; ++b) {
        double d[8], e2[8];                             // (rows beyond the matrix read padding, forwards, or row 0, backwards; nothing is kept)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = 8 * b + u;
          d[u] = te[down ? max(n - 1 - i, 0) : i].x - lm;
          e2[u] = te[down ? max(n - i, 0) : i].y;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const double pn = fma(d[u], p, -e2[u] * pm);
          d[u] = pn * rcp_cubic(p + 1e-290);
          pm = p; p = pn;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int i = 8 * b + u;
          if (i < n) D[(down ? n - 1 - i : i) * P] = d[u];
        }
        const int big = max(__double2hiint(p) & 0x7FF00000, __double2hiint(pm) & 0x7FF00000);
        const double sc = __hiloint2double(0x7FE00000 - big, 0);
        p *= sc; pm *= sc;
      }
    }
    bar();
    {
      // twist where |gamma| is least: z = 1 there, the other entries are products of e / pivot outwards from it
      const int e = tid >> 2, s = tid & 3;
      const double lm = lam[e];
      double best = 1e300, du[2 * NT8], dd[2 * NT8];
      int at = 0;
#pragma unroll
      for (int t = 0; t < 2 * NT8; ++t) { du[t] = Dp[(s + 4 * t) * P + e]; dd[t] = Z[(s + 4 * t) * P + e]; }
#pragma unroll
      for (int t = 0; t < 2 * NT8; ++t) {
        const int i = s + 4 * t;
        const double gamma = fabs(du[t] + dd[t] - (te[i].x - lm));
        if (i < n && gamma < best) { best = gamma; at = i; }
      }
#pragma unroll
      for (int o = 2; o > 0; o >>= 1) {
        const double other = __shfl_xor_sync(0xFFFFFFFFu, best, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, at, o);
        if (other < best || (other == best && oi < at)) { best = other; at = oi; }
      }
      if (s == 0) order[e] = at;
#pragma unroll
      for (int t = 0; t < 2 * NT8; ++t) {
        const int i = s + 4 * t;
        const double f = eo[i < at ? i : max(i - 1, 0)] * rcp_cubic((i < at ? du[t] : dd[t]) + 1e-60);
        Z[i * P + e] = i < n ? (i == at ? 1.0 : -f) : 0.0;
      }
    }
    bar();
    {                                                   // two threads per vector, by whole warps
      const int e = tid >> 1, step = tid & 1 ? 1 : -1;
      double f = 1.0, zz = tid & 1 ? 0.0 : 1.0;
      int i = e < n ? order[e] + step : -1;
      while (i >= 0 && i < n) {                         // four at a time, the loads ahead of the products
        double m[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { const int at = i + u * step; m[u] = at >= 0 && at < n ? Z[at * P + e] : 0.0; }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int at = i + u * step;
          f *= m[u];
          zz = fma(f, f, zz);
          if (at >= 0 && at < n) Z[at * P + e] = f;
        }
        i += 4 * step;
      }
      zz += __shfl_xor_sync(0xFFFFFFFFu, zz, 1);
      if (step > 0 && e < N8) ys[e] = e < rank ? rsqrt_cubic(zz) : 0.0;         // a dependent column of the factor: no vector
    }
  } else {
    // ---- meanwhile: the reflectors in panels of eight, H_8b ... H_8b+7 = I - V_b^T T_b V_b (T_b: inverse of diag(1 / beta) + the
    // upper triangle of V_b V_b^T), a warp per panel ----
    for (int b = warp - TV / 32; b < NT8; b += (EIG_THREADS - TV) / 32) {
      double acc[2][2] = {};
#pragma unroll
      for (int kk = 0; kk < N8; kk += 4) {
        const bool on = 8 * b + g + 2 < n;
        const double a = on ? V[(8 * b + g) * P + kk + q] : 0.0;
        dmma(acc[(kk >> 2) & 1], a, a);                 // the fragments of V_b and of its transpose hold the same entries
      }
      double* t = Tp + 64 * b;
      t[8 * g + 2 * q] = acc[0][0] + acc[1][0]; t[8 * g + 2 * q + 1] = acc[0][1] + acc[1][1];
      __syncwarp();
      double xcol[8];                                   // column `lane` of the lower triangular inverse: T_b transposed
      if (lane < 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          double sum = 0.0;
#pragma unroll
          for (int k = 0; k < i; ++k) sum = fma(t[8 * i + k], xcol[k], sum);
          const double bt = 8 * b + i + 2 < n ? beta_s[8 * b + i] : 0.0;
          xcol[i] = i == lane ? bt : (i > lane ? -bt * sum : 0.0);
        }
      }
      __syncwarp();
      if (lane < 8)
#pragma unroll
        for (int i = 0; i < 8; ++i) t[8 * lane + i] = xcol[i];                 // T_b[lane][i]
    }
  }
  __syncthreads();
  // ---- back through the panels: a warp per eight vectors, which it holds transposed, Z^T -= (Z^T V_b^T) T_b^T V_b: an accumulator tile
  // (lane: row g, columns 2 q and 2 q + 1) is the left operand of the next product as it stands, its columns taken in the order 2 q, then
  // 2 q + 1, so that nothing but V and T comes from shared memory (with Z there, n = 40: 6300 -> 3000 cycles) ----
  for (int tj = warp; tj < NT8; tj += EIG_THREADS / 32) {
    double z[NT8][2];
#pragma unroll
    for (int t = 0; t < NT8; ++t)
#pragma unroll
      for (int h = 0; h < 2; ++h) z[t][h] = 8 * tj + g < n ? Z[(8 * t + 2 * q + h) * P + 8 * tj + g] : 0.0;     // (vectors beyond the matrix)
    const double rz = ys[8 * tj + g];
    __syncwarp();
#pragma unroll 1
    for (int b = (n - 3) >> 3; b >= 0; --b) {
      const bool on = 8 * b + g + 2 < n, on0 = 8 * b + 2 * q + 2 < n, on1 = 8 * b + 2 * q + 3 < n;
      const double *vr = V + (8 * b + g) * P + 2 * q, *v0 = V + (8 * b + 2 * q) * P + g;
      double acc[2][2] = {}, y[2] = {0.0, 0.0};
#pragma unroll
      for (int t = 0; t < NT8; ++t) {
        const double2 v = on ? *reinterpret_cast<const double2*>(vr + 8 * t) : make_double2(0.0, 0.0);
        dmma(acc[0], z[t][0], v.x);
        dmma(acc[1], z[t][1], v.y);
      }
      const double2 tb = *reinterpret_cast<const double2*>(Tp + 64 * b + 8 * g + 2 * q);
      dmma(y, -(acc[0][0] + acc[1][0]), tb.x);
      dmma(y, -(acc[0][1] + acc[1][1]), tb.y);
#pragma unroll
      for (int t = 0; t < NT8; ++t) dmma(z[t], y[0], on0 ? v0[8 * t] : 0.0);
#pragma unroll
      for (int t = 0; t < NT8; ++t) dmma(z[t], y[1], on1 ? v0[P + 8 * t] : 0.0);
    }
    // normalised, in the order of the factor's rows
#pragma unroll
    for (int t = 0; t < NT8; ++t)
#pragma unroll
      for (int h = 0; h < 2; ++h) Z[pos[8 * t + 2 * q + h] * P + 8 * tj + g] = rz != 0.0 ? z[t][h] * rz : 0.0;  // (z may have overflowed)
  }
  __syncthreads();

  metis_pdl_trigger();                                  // what is left is short, or rare
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
    bool again = false;
    X = U; Wb = W;
    if (attempt == 1) {                                 // the start by way of T had dependent vectors
      orth_only = false;
      constexpr float exit_cos2 = EIG_TIGHT_COS2;
      for (int o = tid; o < (NB - 1) * GROUPS; o += EIG_THREADS) {                  // round-robin tournament of the blocks
        const int step = o / GROUPS, m = o % GROUPS;
        const int a = m == 0 ? 0 : (step + m) % (NB - 1) + 1, b = m == 0 ? step % (NB - 1) + 1 : (step + NB - 1 - m) % (NB - 1) + 1;
        pairs[step][m][0] = (uint8_t)min(a, b); pairs[step][m][1] = (uint8_t)max(a, b);
      }
      for (int o = tid; o < NB * RP; o += EIG_THREADS) {
        const int b = o / RP, r = o % RP;
        Yb[o] = make_float2((float)(Lm[r * P + 2 * b] * y_scale), (float)(Lm[r * P + 2 * b + 1] * y_scale));
      }
      __syncthreads();
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
          if (__any_sync(0xFFFFFFFFu, above && active) && lane == 0) flags[sweep] = 1;
          bar();
          if (!flags[sweep]) break;
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
            inv_s[2 * (2 * m + h) + sub] = v > 0.0 ? rsqrt_cubic(v) : 0.0;
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
    }

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
                const double ro = 0.5 * r * (lam[i] + lam[j]);                     // what orthonormalising alone adds to S_ij
                if (fmax(sv[u][e] * sv[u][e], ro * ro) > 1e-28 * fabs(lam[i] * lam[j])) {    // else orthogonal to FP64 rounding, and stays so
                  if (fabs(a) < 0.0625 * fabs(gap) && fabs(b) < 0.0625 * fabs(gap)) {
                    const double rg = rcp_cubic(gap);
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
        if (attempt == 0) { again = true; break; }        // the FP32 sweeps make another start
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
          const double d = b - a, rh = rsqrt_cubic(fma(4.0 * c, c, d * d));
          const double cc = fma(0.5 * fabs(d), rh, 0.5), rs = rsqrt_cubic(cc);
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
  for (int i = warp; i < n; i += EIG_THREADS / 32)
    for (int j = lane; j < n; j += 32) evecs[perm[i] * n + j] = X[i * P + order[j]];
}

}  // namespace metis_small
