// Reciprocal of a pivot in the float64 factorization.
#pragma once

namespace rbf {

// 1 / d for d in [2^-1000, 2^1000): the hardware's approximation (about 20 bits)
// and one third-order step y (1 + e + e^2), e = 1 - d y (Householder's method
// for the reciprocal).  Its error e^3 is below 2^-57 of the result, so that with
// the last rounding the value is within one unit in the last place.  (The
// language's division is about five more of the 65-cycle float64 instructions
// in each step of the serial chain; it serves the pivots outside the range.)
__device__ __forceinline__ double rcp_pos(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const double e = fma(-d, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// d > 0 lies in that range (an integer test: the float64 pipe is what counts)
__device__ __forceinline__ bool rcp_pos_range(double d) {
  return ((unsigned)__double2hiint(d) >> 20) - 23u < 2000u;  // 23: the exponent field of 2^-1000
}

}  // namespace rbf
