// FP64 reciprocal and reciprocal square root with a short dependent chain.
//
// An FP64 instruction of this GPU has a latency of some 65 cycles, so the dozen
// dependent ones of an IEEE division or square root are what serial FP64 code
// (Householder scalars, Jacobi rotations, pivots) waits for.  Here the hardware's
// 20-bit start value is corrected by one step of third order: with e the
// residual, 1/x = y (1 + e + e^2 + ..), e = 1 - x y, and
// x^-1/2 = y (1 + e/2 + 3 e^2/8 + ..), e = 1 - x y^2 (the binomial series),
// three and four dependent instructions; the cut term is below 2^-57 for a start
// value good to 2^-19.  Largest errors found with random mantissas over the whole
// exponent range: 0.504 ulp for the reciprocal and 0.99 for the inverse square
// root, whose x y is rounded (bounds: 0.6 and 1.1).  Arguments near the ends of the exponent
// range, where the start value or a product would leave it, take the library
// functions.
#pragma once

#include <cuda_runtime.h>

namespace peps {

// 2^-700 < |x| < 2^700
__device__ __forceinline__ bool mid_range(double x) {
  return (unsigned)((__double2hiint(x) & 0x7fffffff) - 0x14300000) < 0x57800000u;
}

__device__ __forceinline__ double quick_rcp(double x) {
  if (!mid_range(x)) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

__device__ __forceinline__ double quick_rsqrt(double x) {
  if (!mid_range(x)) return rsqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

}  // namespace peps
