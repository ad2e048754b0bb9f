// FP64 reciprocal and square root in few operations of GB300's FP64 pipe (2 per SM and clock), where a last-place
// rounding does not matter; roundings to FP32 and comparisons beside that pipe, which a conversion takes for 0.8 of an
// FP64 operation.
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

// x >= 2^-14, x finite
__device__ __forceinline__ bool at_least_2_m14(double x) {
  return (unsigned)(__double2hiint(x) - 0x3f100000) < 0x40e00000u;
}

// (float)x, round to nearest even, on the integer pipe: the 11 exponent bits become 8 (bias 1023 - 127 = 0x380), the
// significand loses 29 bits. Outside FP32's normal range and zero, the conversion itself.
__device__ __forceinline__ float rounded_to_float(double x) {
  const unsigned lo = (unsigned)__double2loint(x), hi = (unsigned)__double2hiint(x), e = hi & 0x7ff00000u;
  if (e - 0x38100000u >= 0x0fd00000u) return ((hi << 1) | lo) == 0u ? __uint_as_float(hi) : (float)x;
  unsigned t = __funnelshift_l(lo, hi, 3) - 0xc0000000u;  // exponent and the 23 significand bits that stay
  if ((lo & 0x1fffffffu) + (t & 1u) > 0x10000000u) t += 1u;
  return __uint_as_float(t | (hi & 0x80000000u));
}

// h = (float)x and l = (float)(x - h): the bits that h drops (or lacks, where it was rounded up) are an integer of at
// most 29 bits in units of x's last place. Below 2^-74, where l could be subnormal, in FP64.
__device__ __forceinline__ void split_to_floats(double x, float& h, float& l) {
  const unsigned lo = (unsigned)__double2loint(x), hi = (unsigned)__double2hiint(x), e = hi & 0x7ff00000u;
  if (e - 0x3b500000u >= 0x0c900000u) {
    h = (float)x;
    l = (float)(x - (double)h);
    return;
  }
  unsigned t = __funnelshift_l(lo, hi, 3) - 0xc0000000u;
  int r = (int)(lo & 0x1fffffffu);
  if ((unsigned)r + (t & 1u) > 0x10000000u) {
    t += 1u;
    r -= 0x20000000;
  }
  if ((int)hi < 0) r = -r;
  h = __uint_as_float(t | (hi & 0x80000000u));
  l = __int2float_rn(r) * __uint_as_float(((e >> 20) - 948u) << 23);  // 2^(exponent of x - 52)
}

}  // namespace emppp
