// FP64 reciprocal and square root in a handful of dependent operations, for the
// inner loops in which an FP64 division or library root would be the longest
// chain (a dependent FP64 operation waits about a hundred cycles here, and one
// takes the FP64 pipe the time of about 60 FP32 ones).  Each starts from the
// hardware's approximate instruction (about 20 bits) and takes one step of a
// published iteration of third order, so that what is left of the seed's error is
// below 2^-57: within one unit in the last place (2^-52) of the exact value.
#pragma once

#include <cuda_runtime.h>

namespace rexi {

__device__ __forceinline__ double rcp_seed(double d) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
  return r;
}

// 1 / x for normal x with a normal reciprocal: the hyperpower iteration of order
// three (M. Altman, Pacific J. Math. 10, 1960), r0 (1 + e + e^2) with
// e = 1 - x r0: the geometric series of 1 / x = r0 / (1 - e), e^3 left over.
__device__ __forceinline__ double rcp64(double x) {
  const double r0 = rcp_seed(x);
  const double e = fma(-x, r0, 1.0);
  return fma(r0, fma(e, e, e), r0);
}

// (sqrt(w), 1 / sqrt(w)) for w in (1e-280, 1e280).  The reciprocal root by
// Householder's iteration of order three (A. S. Householder, The Numerical
// Treatment of a Single Nonlinear Equation, 1970), y0 (1 + e/2 + 3 e^2 / 8) with
// e = 1 - w y0^2: the binomial series of (1 - e)^(-1/2), 5 e^3 / 16 left over.
// The root w y by one Newton step (Heron's rule) on s^2 = w with that y for 1 / s.
__device__ __forceinline__ double2 sqrt_rsqrt64(double w) {
  double y0;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y0) : "d"(w));
  const double e = fma(-w * y0, y0, 1.0);
  const double y = fma(y0 * e, fma(0.375, e, 0.5), y0);
  const double s = w * y;
  return make_double2(fma(fma(-s, s, w), 0.5 * y, s), y);
}

}  // namespace rexi
