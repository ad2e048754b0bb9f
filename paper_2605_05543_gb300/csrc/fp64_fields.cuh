// The fields of one pair in FP64, from the source's line at t_n: shared by the FP64 pair kernel (where the forms are
// derived) and the evaluation without device allocation, so that both give the same values. Sums run without the
// electron's charge constant -e / (4 pi eps0) and over c^2 B; both are scaled once per target.
#pragma once

#include "emppp_internal.cuh"
#include "fp64_roots.cuh"

namespace emppp {

// -e / (4 pi eps0)
constexpr double kFieldScale = -kQe / (4.0 * kPi * kEps0);

struct FieldSums {
  double E[3] = {0.0, 0.0, 0.0}, B[3] = {0.0, 0.0, 0.0};
};

// X: the target's separation from where the source's line is at t_n; v: the line's velocity
struct Line {
  double X0, X1, X2, v0, v1, v2;
  double C2;  // c^2 - v^2
  __device__ __forceinline__ void set_c2() { C2 = fma(-v0, v0, fma(-v1, v1, fma(-v2, v2, kC * kC))); }
  __device__ __forceinline__ double XX() const { return fma(X2, X2, fma(X1, X1, X0 * X0)); }
  __device__ __forceinline__ double Xv() const { return fma(X2, v2, fma(X1, v1, X0 * v0)); }
};

// Heaviside's field of uniform motion along the line; cwC2 = c w (c^2 - v^2), root of Dh
__device__ __forceinline__ void heaviside_fields(const Line& l, double cwC2, const Root& root, FieldSums& s) {
  const double iD = root.rsqrt();
  const double pref = cwC2 * ((iD * iD) * iD);
  const double E0 = pref * l.X0, E1 = pref * l.X1, E2 = pref * l.X2;
  s.E[0] += E0;
  s.E[1] += E1;
  s.E[2] += E2;
  // c^2 B = v x E
  s.B[0] = fma(l.v1, E2, fma(-l.v2, E1, s.B[0]));
  s.B[1] = fma(l.v2, E0, fma(-l.v0, E2, s.B[1]));
  s.B[2] = fma(l.v0, E1, fma(-l.v1, E0, s.B[2]));
}

// delay t_n - t_r on the line
__device__ __forceinline__ double line_delay(const Line& l, double XX, double Xv, double sq) {
  const double sum = sq + fabs(Xv);
  const bool pos = __double2hiint(Xv) >= 0;
  return (pos ? sum : XX) * recip_refined(pos ? l.C2 : sum);
}

// retarded velocity and delay of a bracketed pair
struct Retarded {
  double tau, v0, v1, v2;
};

// Lienard-Wiechert fields of a bracketed pair: T1 = t_n - t1, idt = 1 / (t2 - t1), (u0, u1, u2) the newer node's
// velocity, cw = c w. False (nothing added) for coincident particles.
__device__ __forceinline__ bool bracket_fields(const Line& l, double XX, double Xv, const Root& root, double T1,
                                               double idt, double u0, double u1, double u2, double cw, FieldSums& s,
                                               Retarded& out) {
  const double sq = root.sqrt();
  const double tau = line_delay(l, XX, Xv, sq);
  const double f = (T1 - tau) * idt;                                                            // (t_r - t1) / (t2 - t1)
  const double g0 = u0 - l.v0, g1 = u1 - l.v1, g2 = u2 - l.v2;                                  // v2 - v1
  const double e0 = fma(l.v0, tau, l.X0), e1 = fma(l.v1, tau, l.X1), e2 = fma(l.v2, tau, l.X2);  // eta
  const double v0 = fma(f, g0, l.v0), v1 = fma(f, g1, l.v1), v2 = fma(f, g2, l.v2);
  const double eg = fma(e2, g2, fma(e1, g1, e0 * g0));
  const double kappa = fma(-f, eg, sq);
  out = Retarded{tau, v0, v1, v2};
  if (!positive_normal(kappa)) return false;
  const double c2mv2 = fma(-v0, v0, fma(-v1, v1, fma(-v2, v2, kC * kC)));
  const double ik = recip_refined(kappa);
  const double s3 = cw * (ik * ik);                   // c w / kappa^2
  const double s1 = (s3 * ik) * fma(idt, eg, c2mv2);  // c w A / kappa^3
  const double s2 = s3 * idt;
  const double H0 = fma(s1, v0, s2 * g0), H1 = fma(s1, v1, s2 * g1), H2 = fma(s1, v2, s2 * g2);
  s.E[0] = fma(s1, e0, fma(-tau, H0, s.E[0]));
  s.E[1] = fma(s1, e1, fma(-tau, H1, s.E[1]));
  s.E[2] = fma(s1, e2, fma(-tau, H2, s.E[2]));
  s.B[0] = fma(H1, e2, fma(-H2, e1, s.B[0]));
  s.B[1] = fma(H2, e0, fma(-H0, e2, s.B[1]));
  s.B[2] = fma(H0, e1, fma(-H1, e0, s.B[2]));
  return true;
}

}  // namespace emppp
