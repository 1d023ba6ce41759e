// Reciprocals and roots in FP64 for serial chains: the device's approximate instruction and one step of
// Householder's method of order 2 (the residual's series to its second term).
//
//   1 / x:        r with e = 1 - x r;    1 / x = r / (1 - e) = r (1 + e + e^2) + O(r e^3)
//   1 / sqrt(x):  r with e = 1 - x r^2;  r (1 - e)^(-1/2) = r (1 + e / 2 + 3 e^2 / 8) + O(r e^3)
//   sqrt(x):      from r = 1 / sqrt(x), q = x r and one step of Heron's method, q + (x - q^2) r / 2
//
// Error: an approximation good to 2^-19 (e below 2^-18 for the root) leaves terms of at most 2^-57 and
// 2^-56 of the result.  The reciprocal's residual is exact but for one rounding of its own size, so its
// result is off by its last rounding and 1/16 of a unit; the root's residual contains the rounding of x r,
// 2^-53 halved, so its result is off by one unit and a quarter at most; Heron's step squares what r and q
// are off by, so sqrt is off by its last rounding alone (tests/test_gpu_recip.py compares all three with
// quadruple precision and with the ordinary operations).
//
// Why: the serial steps of the dense solver wait for these, three or four dependent operations of 64
// cycles where a correctly rounded division takes about ten (tridiagonalisation and inverse iteration of
// order 564, with the other changes to those steps: 7.5 -> 6.1 and 2.1 -> 0.8 ms).
#pragma once

namespace kss {

// 2^-927 <= |x| < 2^913: what the approximate instructions and the products above stay in range for; other
// arguments (zeros, subnormal and infinite ones among them) take the ordinary operations.
__device__ __forceinline__ bool mid_range(double x) {
  const unsigned e = (unsigned)__double2hiint(x) & 0x7ff00000u;
  return e - 0x06000000u < 0x73000000u;
}
__device__ __forceinline__ double fast_rcp(double x) {
  if (!mid_range(x)) return 1.0 / x;
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double fast_rsqrt(double x) {  // x >= 0
  if (!mid_range(x)) return 1.0 / sqrt(x);
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}
// sqrt(x) from r = fast_rsqrt(x)
__device__ __forceinline__ double sqrt_from(double x, double r) {
  if (!mid_range(x)) return sqrt(x);
  const double q = x * r;
  return fma(fma(-q, q, x), 0.5 * r, q);
}

}  // namespace kss
