// Reciprocal and reciprocal square root in FP64, from the hardware's
// approximations (about 20 bits) by one step of Householder's method of third
// order (A. S. Householder, The Numerical Treatment of a Single Nonlinear
// Equation, 1970): the series of 1 / (1 - e) and (1 - e)^(-1/2) to the second
// power of the approximation's error e.  What is left out, of order e^3, is
// below 2^-59.  An FP64 instruction of a warp holds its sub-partition's FP64
// unit for ~64 cycles; one such step takes fewer of them than second-order
// (Newton) steps, or than a division or a square root.
#pragma once

namespace hz {

// 1 / x for normal x with a normal reciprocal: within 1.1 2^-53 of it
__device__ __forceinline__ double recip3(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1 / sqrt(x) for normal x > 0: within 1.75 2^-53 of it
__device__ __forceinline__ double rsqrt3(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x * y, y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}

}  // namespace hz
