// FP32 shadow record of one history slot, used by the mixed-precision pair path and by the FP32
// delay guess. Three float4 per (particle, slot):
//   q0 = (hi.x, hi.y, hi.z, 1/gamma^2)   hi = fl32(w - origin)
//   q1 = (lo.x, lo.y, lo.z, dev)         lo = fl32((w - origin) - hi), so hi + lo carries ~48 bits; dev: 1.03 times
//                                        the next slot's distance from this slot's line (kNewerMargin), +inf
//                                        until that slot is written
//   q2 = (dbeta.x, dbeta.y, dbeta.z, gamma^2)  dbeta = v/c - beta_ref
// 1/gamma^2 = 1 - beta^2 is formed in FP64, so the FP32 path never subtracts beta^2 from 1. Velocities
// are stored relative to a reference velocity beta_ref (the velocity of one particle of the bunch when
// the state was set): the spread of a bunch's velocities is small, so the FP32 difference of two stored
// velocities (the acceleration of eq:linear) keeps its relative precision; beta itself is
// beta_ref + dbeta.
#pragma once

#include "emppp_internal.cuh"
#include "fp64_roots.cuh"

namespace emppp {

__device__ __forceinline__ void shadow_record(const double origin[3], const double beta_ref[3], double w0, double w1,
                                              double w2, double v0, double v1, double v2, double gamma2, double inv_gamma2,
                                              float4 q[3]) {
  const double ic = 1.0 / kC;
  split_to_floats(w0 - origin[0], q[0].x, q[1].x);
  split_to_floats(w1 - origin[1], q[0].y, q[1].y);
  split_to_floats(w2 - origin[2], q[0].z, q[1].z);
  q[0].w = rounded_to_float(inv_gamma2);
  q[1].w = __int_as_float(0x7f800000);
  q[2] = make_float4(rounded_to_float(v0 * ic - beta_ref[0]), rounded_to_float(v1 * ic - beta_ref[1]),
                     rounded_to_float(v2 * ic - beta_ref[2]), rounded_to_float(gamma2));
}

__device__ __forceinline__ void shadow_record(const double origin[3], const double beta_ref[3], double w0, double w1,
                                              double w2, double v0, double v1, double v2, double gamma2, float4 q[3]) {
  shadow_record(origin, beta_ref, w0, w1, w2, v0, v1, v2, gamma2, 1.0 / gamma2, q);
}

// dev of a slot at w0 with velocity v0 (inv_gamma2: 1 - v0.v0 / c^2) whose next slot, dt later, is at w1 (rounded up: the
// FP32 norm is within 4u, and the added 1e-20 m covers squares that underflow)
__device__ __forceinline__ float line_deviation(double w00, double w01, double w02, double v00, double v01, double v02,
                                                double w10, double w11, double w12, double dt, double inv_gamma2) {
  static_assert(kDevGamma2 == 16384.0, "the comparison below");
  const float d0 = rounded_to_float((w10 - w00) - v00 * dt), d1 = rounded_to_float((w11 - w01) - v01 * dt),
              d2 = rounded_to_float((w12 - w02) - v02 * dt);
  const float up = fmaf(sqrtf(d0 * d0 + d1 * d1 + d2 * d2), 1.0302f, 1e-20f);
  return at_least_2_m14(inv_gamma2) ? up : __int_as_float(0x7f800000);
}
__device__ __forceinline__ float line_deviation(double w00, double w01, double w02, double v00, double v01, double v02,
                                                double w10, double w11, double w12, double dt) {
  return line_deviation(w00, w01, w02, v00, v01, v02, w10, w11, w12, dt,
                        1.0 - (v00 * v00 + v01 * v01 + v02 * v02) * (1.0 / (kC * kC)));
}

// gamma^2 of a stored velocity: 1 / (1 - v.v / c^2)
__device__ __forceinline__ double gamma2_of_v(double v0, double v1, double v2) {
  return 1.0 / (1.0 - (v0 * v0 + v1 * v1 + v2 * v2) / (kC * kC));
}

// Its inverse and gamma^2 as an FP32 record holds them, without the three divisions: the same FP32 values as 1 / g and g
// = gamma2_of_v. The rounded constant 1 / c^2, the quotient and the difference move 1 - v.v / c^2 by at most 2.5 * 2^-53, 2.5
// gamma^2 ulps of it and of its reciprocal, to which recip_refined and the divisions add four; FP32 rounds both ways to
// the same value unless they lie that near the middle of two FP32 values, where the divisions decide (and for |v| >= c).
__device__ __forceinline__ void record_gamma2(double v0, double v1, double v2, double& gamma2, double& inv_gamma2) {
  const double vv = v0 * v0 + v1 * v1 + v2 * v2;
  inv_gamma2 = fma(-vv, 1.0 / (kC * kC), 1.0);
  gamma2 = recip_refined(inv_gamma2);
  const float g = rounded_to_float(gamma2);
  const unsigned near = 8u + 4u * (unsigned)fminf(g, 6e7f);
  auto near_middle = [&](double x) { return ((unsigned)__double2loint(x) & 0x1fffffffu) - (0x10000000u - near) <= 2u * near; };
  if (!positive_normal(inv_gamma2) || g > 6e7f || near_middle(gamma2) || near_middle(inv_gamma2)) {
    gamma2 = gamma2_of_v(v0, v1, v2);
    inv_gamma2 = 1.0 / gamma2;
  }
}

// gamma^2 of a proper velocity: 1 + u.u / c^2 (no cancellation)
__device__ __forceinline__ double gamma2_of_u(double u0, double u1, double u2) {
  return 1.0 + (u0 * u0 + u1 * u1 + u2 * u2) / (kC * kC);
}

// Uniform-motion guess of the older bracket node: the source at its present record (q0n, q2n)
// keeps its velocity; c (t - t_r) = [d.beta + sqrt((d.beta)^2 + (1 - beta^2) d^2)] / (1 - beta^2),
// d = r - w_n. Returns an offset in the window of nw slots, clamped to [0, nw - 2] (requires nw > 1).
__device__ __forceinline__ int uniform_motion_guess(float r0, float r1, float r2, float4 q0n, float4 q2n, float3 bref,
                                                    float inv_cdt, int nw) {
  const float d0 = r0 - q0n.x, d1 = r1 - q0n.y, d2 = r2 - q0n.z;
  const float db = d0 * (bref.x + q2n.x) + d1 * (bref.y + q2n.y) + d2 * (bref.z + q2n.z);
  const float dd = d0 * d0 + d1 * d1 + d2 * d2;
  const float ctau = (db + sqrtf(fmaxf(db * db + q0n.w * dd, 0.f))) * q2n.w;
  const float steps = floorf(ctau * inv_cdt);
  return max(nw - 2 - (int)fminf(fmaxf(steps, 0.f), 1e9f), 0);
}

}  // namespace emppp
