// FP64 reciprocal and square root in few operations of GB300's FP64 pipe (2 per SM and clock), where a last-place
// rounding does not matter.
#pragma once

namespace emppp {

// 1 / x for finite x > 0: the hardware's approximate reciprocal y (about 2^-20 relative) refined by one
// step of Householder's third-order iteration, y <- y + y (e + e^2) with e = 1 - x y, which leaves e^3: three
// FP64-pipe operations (two Newton-Raphson steps, as before, took four). Within a few units in the last
// place, not correctly rounded.
__device__ __forceinline__ double recip_refined(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// The same iteration for the root: with y the hardware's approximation of 1 / sqrt(x), t = x y and
// e = 1 - x y^2, sqrt(x) = t / sqrt(1 - e) = t + t e (1/2 + 3/8 e) + O(e^3), and 1 / sqrt(x) likewise from y.
// Both share t, e and the bracket; each costs two more operations.
struct Root {
  double y, t, e, q;
  __device__ __forceinline__ explicit Root(double x) {
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    t = x * y;
    e = fma(-t, y, 1.0);
    q = fma(e, 0.375, 0.5);
  }
  __device__ __forceinline__ double sqrt() const { return fma(t * e, q, t); }
  __device__ __forceinline__ double rsqrt() const { return fma(y * e, q, y); }
};

// finite, positive and normal, decided on the high word: a comparison of doubles would take the FP64 pipe
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)(__double2hiint(x) - 0x00100000) < 0x7fe00000u;
}

}  // namespace emppp
