// 1/x and 1/sqrt(x) in FP64 for the dense kernels of a decomposition, which take them by the eight in unrolled loops.
#pragma once

namespace metis_small {

// Newton-Raphson on f(y) = 1/y - x and on f(y) = 1/y^2 - x, two steps from the hardware's approximation:
//   y <- y + y (1 - x y)             1 - x y' = (1 - x y)^2
//   y <- y + y (1/2 - x/2 y y)       1 - x y'^2 = 3/4 r^2 + r^3/4,  r = 1 - x y^2
// so a seed good to 2^-15 leaves rounding alone: 2^-53 (1 + 2^-20) of the value for the reciprocal; 1.5 x 2^-53 (1 + 2^-20) for the root, whose
// product x/2 y is rounded too.  For normal x whose result is normal; zero, infinities and subnormals give NaNs or infinities, and no caller uses them.
// (1.0 / x and rsqrt(x), whose branch for such x keeps neighbours of a loop from running side by side: forward of 1024 tokens 192 -> 197 us,
// the LLaMA-3-8B q_proj step 687 -> 703 us.)
__device__ __forceinline__ double rcp_newton(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(y, fma(-x, y, 1.0), y);
  return y;
}
__device__ __forceinline__ double rsqrt_newton(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int i = 0; i < 2; ++i) y = fma(y, fma(-0.5 * x * y, y, 0.5), y);
  return y;
}

}  // namespace metis_small
