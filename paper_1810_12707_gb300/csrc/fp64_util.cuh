// fp64_util.cuh -- FP64 reciprocal, quotient and square root in few FP64 instructions, for kernels
// that the FP64 pipe bounds (1.7 fused multiply-adds per clock and SM on GB300).  Each starts from the
// hardware's approximation (relative error e of about 2^-20) and takes one step of Householder's
// third-order iteration, whose remaining error, of order e^3, is below 2^-57, with the residual in a
// fused multiply-add: only the last one rounds.  Largest errors over 200,000 random arguments each, in
// units in the last place: reciprocal 0.502, quotient 0.500 (every one the rounded quotient), root 0.510.
#pragma once

#include <cuda_runtime.h>

namespace mhd {

// 1 / x = r (1 + e + e^2), e = 1 - x r: four instructions, about half a division's.  A NaN for x = 0
// and x infinite.
__device__ __forceinline__ double rcp3(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// Whether x is a normal, positive or negative, finite number whose reciprocal is one too.
__device__ __forceinline__ bool rcp3_covers(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return h - 0x00200000u < 0x7fa00000u;
}
// 1 / x for every x: the flux pass's, whose densities may be anything.
__device__ __forceinline__ double rcp_any(double x) {
  if (rcp3_covers(x)) return rcp3(x);
  return 1.0 / x;
}
// m / x with r = 1 / x from rcp3: the quotient m r corrected by its remainder (Markstein), which
// rounds correctly but for rare cases (|m| above 2^-960, or the remainder may be subnormal).  Three
// instructions.  An infinite m r is the quotient: its remainder would be infinite too, and their sum a
// NaN.
__device__ __forceinline__ double quotient(double m, double x, double r) {
  const double q = m * r;
  const double c = fma(fma(-x, q, m), r, q);
  return (__double2hiint(q) & 0x7ff00000) == 0x7ff00000 ? q : c;
}

// sqrt(x) = s (1 + e/2 + 3 e^2 / 8), s = x y, e = 1 - s^2 / x, y the approximate 1 / sqrt(x): the
// leading term s e / 2 as (x - s^2) y / 2, so that the rounding of s drops out (taken from 1 - s y, an
// instruction less, half of it stayed in the result: 0.75 units in the last place).  Six instructions.
// Numbers below 2^-959, whose x - s^2 may be subnormal, and zero, negative, infinite and NaN
// arguments take the library's root.
__device__ __forceinline__ double sqrt3(double x) {
  if ((unsigned)__double2hiint(x) - 0x04000000u >= 0x7bf00000u) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double s = x * y, e = fma(-s, y, 1.0);
  return fma(fma(-s, s, x) * y, fma(0.375, e, 0.5), s);
}

}  // namespace mhd
