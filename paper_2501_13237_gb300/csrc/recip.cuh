// Reciprocals and reciprocal square roots from the hardware's estimate y and the binomial
// series of the remaining factor: with r = 1 - x y, 1 / x = y (1 - r)^-1 = y (1 + r + r^2 +
// ...); with r = 1 - x y^2, 1 / sqrt(x) = y (1 - r)^(-1/2) = y (1 + r / 2 + 3 r^2 / 8 + 5 r^3 / 16
// + ...).  Cut after r they are Newton's steps.  A divide or square root costs several times
// their instructions, which in float64 (64 cycles each for a warp) stand on every row and
// column of the factorisations.
#pragma once
#include "common.cuh"

namespace nne {

// 1 / x, x normal and finite: estimate of 20 bits, cut after r^2, so r^3 = 2^-60 before the
// last rounding; relative error at most 1.1 x 2^-53.
__device__ __forceinline__ double rcp_series(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double r = fma(-x, y, 1.0);
  return fma(y, fma(r, r, r), y);
}

// 1 / sqrt(x), x > 0: estimate of 2 ulp, cut after r; relative error at most 2^-23.
__device__ __forceinline__ float rsqrt_series(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);
}
// x normal and finite: estimate of 20 bits, whose square is exact, cut after r^3, so r^4 = 2^-76
// before the last rounding; relative error at most 1.1 x 2^-53.
__device__ __forceinline__ double rsqrt_series(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double r = fma(-x, y * y, 1.0);   // (-x * y) * y would round the product first: 1.3 x 2^-53
  return fma(y * r, fma(r, fma(r, 0.3125, 0.375), 0.5), y);
}

}  // namespace nne
