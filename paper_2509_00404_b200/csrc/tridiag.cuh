// Symmetric eigenproblems by way of a tridiagonal matrix, FP64: Householder reduction, eigenvalues by multisection with Sturm
// counts, eigenvectors by twisted factorisations.  What it returns is the start of a refinement (small_eig.cuh, bigrank.cuh)
// and not a result: vectors of eigenvalues that agree to 1e-9 or so come out linearly dependent, and the caller has to look.
#pragma once
#include "common.cuh"
#include "reciprocal.cuh"

namespace metis_tri {

// The reflector that takes x (first entry x0, squared length sq) to alpha e_1: H = I - beta v v^T, v = x - alpha e_1.
// x whose square is below rounding of a matrix with entries near one is left alone (beta = 0).
__device__ __forceinline__ void reflector(double x0, double sq, double& alpha, double& beta) {
  const double len = sq * metis_small::rsqrt_newton(sq);
  const bool on = sq > 1e-60;
  alpha = on ? -copysign(len, x0) : x0;
  beta = on ? metis_small::rcp_newton(fma(fabs(x0), len, sq)) : 0.0;
}

// Sturm sequences of T - x over 8 * blocks rows for M points x: the numbers of eigenvalues below them.  te[i] = (d_i, e_{i-1}^2),
// e_{-1} = 0, squares not zero elsewhere; rows beyond the matrix hold (large, 0).  p_{i+1} = (d_i - x) p_i - e_{i-1}^2 p_{i-1} without
// a division is one multiply-add deep per row; eight rows change a value by at most 2^+-480, after which both are scaled by
// the same power of two.  A row's 16 bytes cost a warp four cycles of the shared-memory pipe, its six instructions of two points
// twelve to twenty of the FP64 pipe.
template <int M>
__device__ __forceinline__ void sturm_counts(const double2* te, int blocks, const double (&x)[M], int (&count)[M]) {
  double pm[M], p[M];
  unsigned int signs[M];
#pragma unroll
  for (int u = 0; u < M; ++u) { pm[u] = 0.0; p[u] = 1.0; signs[u] = 0u; count[u] = 0; }
#pragma unroll 1
  for (int b = 0; b < blocks; ++b) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const double2 t = te[8 * b + i];
#pragma unroll
      for (int u = 0; u < M; ++u) {
        const double next = fma(t.x - x[u], p[u], -t.y * pm[u]);
        pm[u] = p[u]; p[u] = next;
        signs[u] = __funnelshift_l((unsigned int)__double2hiint(next), signs[u], 1);
      }
    }
#pragma unroll
    for (int u = 0; u < M; ++u) {
      count[u] += __popc((signs[u] ^ (signs[u] >> 1)) & 0xFFu);
      const double f = __hiloint2double(0x7FE00000 - max(__double2hiint(p[u]) & 0x7FF00000, __double2hiint(pm[u]) & 0x7FF00000), 0);
      p[u] *= f; pm[u] *= f;
    }
  }
}

// Eigenvalue number `below` (counted upwards from zero) of T, by L lanes of a warp whose 32 lanes all call (lanes L i ... L i + L - 1;
// what is left over repeats the last group's work): every round splits the interval of bit patterns (the logarithm of the
// value, nearly) into 2 L + 1, two points per lane.
template <int L>
__device__ __forceinline__ double multisect(const double2* te, int blocks, long long lo, long long hi, int below, int rounds) {
  constexpr int PARTS = 2 * L + 1, GROUPS = 32 / L;
  const int lane = threadIdx.x & 31, grp = min(lane / L, GROUPS - 1), s = min(lane - L * grp, L - 1);
#pragma unroll 1
  for (int r = 0; r < rounds; ++r) {
    const long long w = (long long)((unsigned long long)(hi - lo + PARTS - 1) / PARTS), at = lo + w * (s + 1);
    const double x[2] = {__longlong_as_double(at), __longlong_as_double(at + L * w)};
    int c[2];
    sturm_counts<2>(te, blocks, x, c);
    const unsigned int v0 = (__ballot_sync(0xFFFFFFFFu, c[0] > below) >> (L * grp)) & ((1u << L) - 1);
    const unsigned int v1 = (__ballot_sync(0xFFFFFFFFu, c[1] > below) >> (L * grp)) & ((1u << L) - 1);
    const int f = __ffs((int)(v0 | (v1 << L) | (1u << (2 * L)))) - 1;          // the first point above the eigenvalue
    hi = lo + w * (f + 1);
    lo += w * f;
  }
  return __longlong_as_double(lo + ((hi - lo) >> 1));
}

}  // namespace metis_tri
