// Reciprocal square root and reciprocal for the rotation and reflector scalars.
#pragma once

namespace dh2 {

// FP32: the hardware's approximations (a few ulp; the rotations and reflections
// stay unitary to that level).
__device__ __forceinline__ float frsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ float frcp(float x) { return __fdividef(1.f, x); }

// FP64: from an approximation y0 the first terms of the binomial series
//   x^{-1/2} = y0 (1 - h)^{-1/2} = y0 (1 + h/2 + 3/8 h^2 + ...), h = 1 - x y0^2,
//   x^{-1}   = y0 (1 - h)^{-1}   = y0 (1 + h + h^2 + ...),       h = 1 - x y0,
// in 5 and 3 operations of the narrow FP64 pipe.  With y0 off by 2^-19 the terms
// left out are below 2^-55; with h's rounding and the last one the result lies
// within 1 ulp (2 ulp are relied on).  Arguments are normal and finite (squared
// norms above Eps::tiny), or give NaN.
__device__ __forceinline__ double rsqrt_from(double x, double y0) {
  const double h = fma(-x * y0, y0, 1.0);
  return fma(y0 * h, fma(0.375, h, 0.5), y0);
}
__device__ __forceinline__ double frsqrt(double x) {
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
  return rsqrt_from(x, y0);
}
__device__ __forceinline__ double frcp(double x) {
  double y0;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(x));
  const double h = fma(-x, y0, 1.0);
  return fma(y0, fma(h, h, h), y0);
}

}  // namespace dh2
