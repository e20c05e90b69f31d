// fastmath.cuh -- reciprocal for the FP64 transport arithmetic.
//
// rcp_nr(s): one third-order Newton step for 1/s, x (1 + e + e^2) with e = 1 - s x, from the
// hardware's approximate reciprocal (PTX rcp.approx.ftz.f64, relative error below 2^-20, so e^3 is
// below the FP64 rounding): 1 ulp at three FP64 operations, against about eight for an IEEE-rounded
// division.  Valid for normal s (subnormal s flush to zero and give an infinite seed); the
// transport code calls it only with normal, finite arguments.
#pragma once
#include <cuda_runtime.h>

namespace ct {

__device__ __forceinline__ double rcp_nr(double s) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(s));
  const double e = fma(-s, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

}  // namespace ct
