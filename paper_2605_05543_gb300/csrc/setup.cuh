// What the pair kernels need of a step besides the rings: the slot tables and per-source vectors. Formed by the set-up
// launch, or by the post-pair launch of the step before.
#pragma once

#include "emppp_internal.cuh"
#include "fp64_roots.cuh"

namespace emppp {

// Slot-table entry of window offset l (slot p0 + l, modulo D) at time t_n (Sec. 2.2): the squared
// light-travel distance (c (t_n - t_k))^2 in exactly the operation order of the reference evaluation
// (so that the FP64 node test decides identically), its upper guard-band threshold in FP32, c (t_n - t_k) in
// FP32 hi and lo, t_n - t_k and 1 / (t_{k+1} - t_k).
constexpr double kGuardHi = (1.0 + kGuardBand) / (1.0 - kGuardBand);

// FP32 upper threshold of a slot's (c (t_n - t_k))^2 (the node test is true above it)
__device__ __forceinline__ float upper_threshold(double lhs) { return __double2float_ru(lhs * kGuardHi); }

// pn: the present slot, whose time is t_n
__device__ __forceinline__ void slot_table(const DeviceState& s, int l, int p0, int pn, int nwin, double t_n) {
  int p = p0 + l;
  if (p >= s.D) p -= s.D;
  const double tk = p == pn ? t_n : s.slot_t[p];
  const double ct = __dmul_rn(kC, __dsub_rn(t_n, tk));
  const double lhs = __dmul_rn(ct, ct);
  s.tab.lhs64[p] = lhs;
  float icdt = 0.f;
  if (l + 1 < nwin) {
    int q = p + 1 == s.D ? 0 : p + 1;
    const double dtk = (q == pn ? t_n : s.slot_t[q]) - tk;
    const double idt = recip_refined(dtk);
    s.tab.tab64[p] = make_double2(t_n - tk, idt);
    icdt = (float)(idt * (1.0 / kC));
  } else {
    s.tab.tab64[p] = make_double2(t_n - tk, 0.0);
  }
  s.tab.tab32[p] = make_float4(upper_threshold(lhs), (float)(ct - (double)(float)ct), (float)ct, icdt);
}

// the first ten doubles of source j's ext64: present position x, line offset after T0 from slot k0's record, and the four
// values given (the velocity, in units of the path's own, and what follows it)
__device__ __forceinline__ void write_line(const DeviceState& s, long long j, const double* x, const double* r0,
                                           double T0, double e6, double e7, double e8, double e9) {
  double2* e = s.ext64 + (size_t)j * (kExt64 / 2);
  e[0] = make_double2(x[0], x[1]);
  e[1] = make_double2(x[2], fma(r0[3], T0, r0[0] - x[0]));
  e[2] = make_double2(fma(r0[4], T0, r0[1] - x[1]), fma(r0[5], T0, r0[2] - x[2]));
  e[3] = make_double2(e6, e7);
  e[4] = make_double2(e8, e9);
}

// slot k0 of a source: FP64 record, FP32 beta - beta_ref and 1/gamma^2, gamma^2
struct Oldest {
  double r[6];
  float db[3], ig2, gamma2;

  __device__ __forceinline__ void load(const DeviceState& s, SetupExt ext, long long j, int p0) {
    const double2* q = reinterpret_cast<const double2*>(s.rec64 + ((size_t)j * s.D + p0) * 6);
    const double2 a = q[0], b = q[1], c = q[2];
    r[0] = a.x, r[1] = a.y, r[2] = b.x, r[3] = b.y, r[4] = c.x, r[5] = c.y;
    if (ext == SetupExt::mixed) {
      const float4* f = reinterpret_cast<const float4*>(s.rec32 + ((size_t)j * s.D + p0) * 12);
      const float4 q2 = f[2];
      ig2 = f[0].w;
      db[0] = q2.x, db[1] = q2.y, db[2] = q2.z, gamma2 = q2.w;
    }
  }
};

// the FP64 path's vectors of source j, at x at t_n, T0 after slot k0
__device__ __forceinline__ void source_vectors_fp64(const DeviceState& s, long long j, const double* x, const Oldest& o,
                                                    double T0) {
  const double v0 = o.r[3], v1 = o.r[4], v2 = o.r[5];
  const double C2 = fma(-v0, v0, fma(-v1, v1, fma(-v2, v2, kC * kC)));
  const double cw = kC * s.wts[j];
  write_line(s, j, x, o.r, T0, v0, v1, v2, C2);
  s.ext64[(size_t)j * (kExt64 / 2) + 5] = make_double2(cw, cw * C2);
}

// the mixed path's vectors of source j, at x at t_n, T0 after slot k0; seg: the record of slot n - 1, dtl before t_n, or
// nullptr (n = k0)
__device__ __forceinline__ void source_vectors_mixed(const DeviceState& s, long long j, const double* x, const Oldest& o,
                                                     double T0, const double* seg, double dtl) {
  // fast sources: the mixed kernel may need their line in FP64 (kXbGuard)
  if (o.ig2 < kXbGamma)
    write_line(s, j, x, o.r, T0, o.r[3] * (1.0 / kC), o.r[4] * (1.0 / kC), o.r[5] * (1.0 / kC), 0.0);
  float4* ext = s.ext32 + (size_t)j * kExtCount;
  ext[kExtLine] = make_float4(rounded_to_float((o.r[0] + o.r[3] * T0) - x[0]),
                              rounded_to_float((o.r[1] + o.r[4] * T0) - x[1]),
                              rounded_to_float((o.r[2] + o.r[5] * T0) - x[2]), o.gamma2);
  ext[kExtOldest] = make_float4(o.db[0], o.db[1], o.db[2], o.ig2);
  const double c0 = x[0] - o.r[0], c1 = x[1] - o.r[1], c2 = x[2] - o.r[2];
  const double ct = __dmul_rn(kC, T0);
  const double cc = c0 * c0 + c1 * c1 + c2 * c2;
  const double rhs = (double)upper_threshold(__dmul_rn(ct, ct)) * (1.0 + kChordMargin) - cc * (1.0 - kChordMargin);
  ext[kExtChord] = make_float4(rounded_to_float(c0), rounded_to_float(c1), rounded_to_float(c2),
                               seg ? fmaxf(__double2float_ru(rhs), 0.f) : __int_as_float(0x7f800000));
  if (!seg) return;  // no segment [n-1, n] in the window
  const BunchDesc& bd = s.bunches[s.nbunch == 1 ? 0 : s.bunch_of[j]];
  float4 h, l;
  split_to_floats((seg[0] + seg[3] * dtl) - bd.origin[0], h.x, l.x);
  split_to_floats((seg[1] + seg[4] * dtl) - bd.origin[1], h.y, l.y);
  split_to_floats((seg[2] + seg[5] * dtl) - bd.origin[2], h.z, l.z);
  h.w = l.w = 0.f;
  ext[kExtSegHi] = h;
  ext[kExtSegLo] = l;
}

}  // namespace emppp
