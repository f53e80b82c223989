// Symmetric eigenproblems by way of a tridiagonal matrix, FP64: Householder reduction, eigenvalues by multisection with Sturm
// counts, eigenvectors by twisted factorisations.  What it returns is the start of a refinement (small_eig.cuh, bigrank.cuh)
// and not a result: vectors of eigenvalues that agree to 1e-9 or so come out linearly dependent, and the caller has to look.
#pragma once
#include "common.cuh"
#include "reciprocal.cuh"

namespace metis_tri {

// The reflector that takes x (first entry x0, squared length sq) to alpha e_1: H = I - beta v v^T, v = x - alpha e_1.
// x whose square is below rounding of a matrix with entries near one is left alone (beta = 0).
// The length and the reciprocal 1 / (|x0| len + sq) come side by side: the approximation that the root starts from starts the reciprocal too.
__device__ __forceinline__ void reflector(double x0, double sq, double& alpha, double& beta) {
  const double y = metis_small::rsqrt_seed(sq), t = sq * y, seed = metis_small::rcp_seed(fma(fabs(x0), t, sq));
  const double r = fma(-t, y, 1.0), len = fma(t * r, fma(r, 0.375, 0.5), t);
  const bool on = sq > 1e-60;
  alpha = on ? -copysign(len, x0) : x0;
  beta = on ? metis_small::rcp_step(fma(fabs(x0), len, sq), seed) : 0.0;
}

// Squares below this count as it (a square of zero would end a Sturm sequence): the root is a rounding of entries near one.
constexpr double TINY_SQUARE = 0x1p-104;

// Sturm sequences of T - x over 8 * blocks rows for M points x: the numbers of eigenvalues below them.  te[i] = (d_i, e_{i-1}^2),
// e_{-1} = 0, squares at least TINY_SQUARE elsewhere; rows beyond the matrix hold (large, 0), and one more block of anything can be
// read.  p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} without a division is one multiply-add (8 cycles) deep per row; eight rows change
// a value by at most 2^+-440.  A power of two brings both values back near one; it is worked out behind a block and applied behind the
// next, off the chain, and a row's entries are loaded a block ahead.  With a warp on each of the four schedulers two points take 24 cycles a row and 210
// for the rest of a call, one point 19 and 190, two warps with two points each 43.
template <int M>
__device__ __forceinline__ void sturm_counts(const double2* te, int blocks, const double (&x)[M], int (&count)[M]) {
  double pm[M], p[M], f[M];
  unsigned int signs[M];
  double2 t[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) t[i] = te[i];
#pragma unroll
  for (int u = 0; u < M; ++u) { pm[u] = 0.0; p[u] = 1.0; f[u] = 1.0; signs[u] = 0u; count[u] = 0; }
#pragma unroll 1
  for (int b = 0; b < blocks; ++b) {
    te += 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
#pragma unroll
      for (int u = 0; u < M; ++u) {
        const double next = fma(t[i].x - x[u], p[u], -t[i].y * pm[u]);
        pm[u] = p[u]; p[u] = next;
        signs[u] = __funnelshift_l((unsigned int)__double2hiint(next), signs[u], 1);
      }
      t[i] = te[i];
    }
#pragma unroll
    for (int u = 0; u < M; ++u) {
      count[u] += __popc((signs[u] ^ (signs[u] >> 1)) & 0xFFu);
      p[u] *= f[u]; pm[u] *= f[u];
      f[u] = __hiloint2double(0x7FE00000 - max(__double2hiint(p[u]) & 0x7FF00000, __double2hiint(pm[u]) & 0x7FF00000), 0);
    }
  }
}

// Eigenvalue number `below` (counted upwards from zero) of T, by L lanes of a warp whose 32 lanes all call (lanes L i ... L i + L - 1;
// what is left over repeats the last group's work): every round splits the interval of bit patterns (the logarithm of the
// value, nearly) into L M + 1, M points per lane.
template <int L, int M>
__device__ __forceinline__ double multisect(const double2* te, int blocks, long long lo, long long hi, int below, int rounds) {
  constexpr int PARTS = L * M + 1, GROUPS = 32 / L;
  const int lane = threadIdx.x & 31, grp = min(lane / L, GROUPS - 1), s = min(lane - L * grp, L - 1);
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const long long w = (long long)((unsigned long long)(hi - lo + PARTS - 1) / PARTS), at = lo + w * (s + 1);
    double x[M];
    int c[M];
#pragma unroll
    for (int u = 0; u < M; ++u) x[u] = __longlong_as_double(at + L * w * u);
    sturm_counts<M>(te, blocks, x, c);
    unsigned int over = 1u << (L * M);                    // bit b: point b has more than `below` eigenvalues under it
#pragma unroll
    for (int u = 0; u < M; ++u) {
      if (L == 1) over |= c[u] > below ? 1u << u : 0u;
      else over |= ((__ballot_sync(0xFFFFFFFFu, c[u] > below) >> (L * grp)) & ((1u << L) - 1)) << (L * u);
    }
    const int f = __ffs((int)over) - 1;
    hi = lo + w * (f + 1);
    lo += w * f;
  }
  return __longlong_as_double(lo + ((hi - lo) >> 1));
}

}  // namespace metis_tri
