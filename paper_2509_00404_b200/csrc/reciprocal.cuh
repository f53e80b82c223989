// 1/x and 1/sqrt(x) in FP64 for the dense kernels of a decomposition, which take them by the eight in unrolled loops.
#pragma once

namespace metis_small {

// One step of third order from the hardware's approximation:
//   e = 1 - x y,    y <- y (1 + e + e^2)            1 - x y' = e^3
//   r = 1 - x y^2,  y <- y (1 + r / 2 + 3/8 r^2)    1 - x y'^2 = 5/8 r^3 + O(r^4)
// (the first terms of 1 / (1 - e) and of 1 / sqrt(1 - r)).  The seeds are good to 2^-19.9 (reciprocal) and 2^-20 (root: r up to 2^-19), measured over 2^28
// values of a period, so a step leaves rounding alone: 2^-53 (1 + 2^-6) of the value for the reciprocal; 1.5 x 2^-53 (1 + 2^-5) for the root, whose
// product x y is rounded too.  For normal x whose result is normal; zero, infinities and subnormals give NaNs or infinities, and no caller uses them.
// (Two Newton-Raphson steps are eight and sixteen cycles longer, 47 and 63 in all.  1.0 / x and rsqrt(x), whose branch for such x keeps neighbours of a
// loop from running side by side: forward of 1024 tokens 192 -> 197 us, the LLaMA-3-8B q_proj step 687 -> 703 us.)
__device__ __forceinline__ double rcp_seed(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double rsqrt_seed(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
// the reciprocal from an approximation y good to 2^-18
__device__ __forceinline__ double rcp_step(double x, double y) {
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ double rcp_cubic(double x) { return rcp_step(x, rcp_seed(x)); }
__device__ __forceinline__ double rsqrt_cubic(double x) {
  const double y = rsqrt_seed(x), r = fma(-x * y, y, 1.0);
  return fma(y * r, fma(r, 0.375, 0.5), y);
}

}  // namespace metis_small
