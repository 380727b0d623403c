// Reciprocals and square roots of doubles from a single-precision start and two Newton steps (plain scalar
// code; x within the range of a normal float).  sqrt and a division are some twenty dependent FP64
// instructions each, of 64 cycles on this GPU; these are four to six.  The second step adds a correction to
// a number that is right to 2^-44, so that its last sum is what rounds.  Largest errors over 2 10^6 random
// arguments with the start two float ulps off: rsqrt_nr 1.0 ulp (1 / sqrt(x): 1.5), rcp_nr 0.5, sqrt_nr 0.5.
// (With the second step as a product, and x times it for the root: 1.7, 0.5 and 2.8.)
// tests/test_newton_host.py compiles this file for the host.
#pragma once

namespace peps {

// y <- y (3 - x y^2) / 2, then y <- y + y (1 - x y^2) / 2
__device__ __forceinline__ double rsqrt_nr(double x) {
  double y = (double)rsqrtf((float)x);
  y = y * fma(-0.5 * x, y * y, 1.5);
  return fma(0.5 * y, fma(-x * y, y, 1.0), y);
}
// r <- r + r (1 - x r), twice
__device__ __forceinline__ double rcp_nr(double x) {
  double r = (double)__frcp_rn((float)x);
  r = fma(r, fma(-x, r, 1.0), r);
  return fma(r, fma(-x, r, 1.0), r);
}
// sqrt(x), y = rsqrt_nr(x)
__device__ __forceinline__ double sqrt_nr(double x, double y) {
  const double s = x * y;
  return fma(0.5 * y, fma(-s, s, x), s);
}

}  // namespace peps
