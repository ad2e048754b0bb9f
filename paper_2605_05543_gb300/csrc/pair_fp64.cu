// FP64 all-pairs Lienard-Wiechert field evaluation with the retarded-time solve (Sec. 2.1-2.2).
//
// One thread owns one target i (present position r = x_i^n at t = t_n) and walks the sources j of
// its slice. Per pair:
//   1. bracket the retarded time in j's history with the node test
//        P(k):  (c (t - t_k))^2 <= |r - w_{j,k}|^2       (true: t_r at or before t_k)
//      evaluated in FP32 on the shadow ring's hi/lo split against guard-band thresholds of the slot
//      tables, and in FP64 in the reference operation order between them (so decisions agree bit for
//      bit): out-of-history if P(k0), near-field shortcut if not P(n-1), else bisection (Sec. 2.2);
//      or, with the closed-form proposal, a guarded galloping search started at the slot predicted
//      by uniform motion from j's present state. Both return the unique sign change of P.
//   2. linear reconstruction (eq:dt, eq:linear): delta t from the quadratic, w = w1 + v1 dt,
//      v = v1 + (dt / (t2 - t1)) (v2 - v1), a = (v2 - v1) / (t2 - t1); or, in the comparison variant MID,
//      the bracket's midpoint values of eq:mid.
//   3. Lienard-Wiechert E (eq:LW_E) and B = eta_hat x E / c (eq:LW_B), summed over j != i in
//      blocks of kTile sources (blocked summation keeps the FP64 rounding error of a 65536-term
//      sum near 1e-14 of the sum of magnitudes).
//   Out of history (eq:linear2) the source moves uniformly with v1 along the line through w_{k0}, and its
//   Lienard-Wiechert field is Heaviside's field about the line's point at t_n: with X = r - w_{k0} -
//   v1 (t_n - t_{k0}), E = kq c (c^2 - v1^2) X / [|X|^2 (c^2 - v1^2) + (X.v1)^2]^{3/2}, B = v1 x E / c^2.
//   It is the same field, without the retarded reconstruction. How 2. and 3. are formed: at the kernel.
// Targets are taken in the spatial order of order.cu (when given), so that the pairs of a warp mostly
// take the same branch; which thread evaluates a target does not change its result.
// The arithmetic is FP64-pipe bound (GB300: 2 DFMA/clk/SM); everything that is not an FP64 result
// (the guess, the node tests outside the guard band, indices, loads) runs on the FP32/INT pipes beside it.
#include "../../include/emppp.h"
#include "emppp_internal.cuh"
#include "fp64_fields.cuh"
#include "mlp.cuh"
#include "shadow.cuh"

namespace emppp {

namespace {

struct PairArgs {
  const double* __restrict__ rec64;
  const float* __restrict__ rec32;
  const double* __restrict__ lhs64;
  const float4* __restrict__ tab32;  // per slot: FP32 upper guard-band threshold of (c (t_n - t_k))^2
  const double2* __restrict__ tab64;  // per slot: t_n - t_k, 1 / (t_{k+1} - t_k)
  const double2* __restrict__ ext64;  // [N][kExt64 / 2] per source (ring.cu)
  const StepState* __restrict__ state;
  double* __restrict__ out;  // [S][N][6] (S = 1: [N][6] temporary) -- see launch
  double* __restrict__ E;
  double* __restrict__ B;
  unsigned long long* stats;
  int* err;
  long long N;
  int D;
  int nbunch;
  const BunchDesc* __restrict__ bunches;
  const BunchSched* __restrict__ sched;
  int nitems;  // work items of all bunches
  int* work;   // work-item counter (zero at launch)
  const mlp::InferImage* __restrict__ net;  // proposal network, inference form (EMPPP_PROPOSAL_MLP)
  unsigned long long* scale;  // adaptive time step: eta_min / v_max^2 reduction
  double eta_allow;
  const int* __restrict__ order;  // spatial order of the targets (nullptr: index order)
  int* __restrict__ dump;  // [N][N] bracket of every evaluated pair, 4 (k1 - k0) + branch (DUMP instances only)
};

// node test P(k) with the reference operation order (no contraction)
__device__ __forceinline__ bool node_test(double r0, double r1, double r2, const double* __restrict__ w,
                                          double lhs) {
  const double d0 = __dsub_rn(r0, __ldg(w + 0));
  const double d1 = __dsub_rn(r1, __ldg(w + 1));
  const double d2 = __dsub_rn(r2, __ldg(w + 2));
  const double rhs = __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
  return lhs <= rhs;
}

struct Window {
  int p0, D, nw;  // slots of the usable window k0..n are addressed by their offset l = k - k0 (0..nw-1)
  int* err;       // device error word (the debug build's range checks)
  __device__ __forceinline__ int phys(int l) const {
    const int p = p0 + debug_index(l, 0, nw, err);
    return p >= D ? p - D : p;
  }
};

// sources staged in shared memory at a time, and the pairs of one partial sum
constexpr int kTile = 64;

}  // namespace

// What bounds it: the FP64 pipe, 2 operations per SM and clock, so that a warp instruction holds it for 16
// cycles. Everything else (guess, node tests, indices, loads) runs beside it; the kernel's cost is its count of
// FP64 operations, about 33 for a pair beyond the history and 72 for one inside it:
//   - both start from X, the target's separation from where the source's line w1 + v1 (t' - t1) is at t_n, and
//     from Dh = |X|^2 (c^2 - v1^2) + (X.v1)^2, a sum of non-negative terms. Out of history Heaviside's field
//     follows at once. Inside it tau = t_n - t_r is the positive root of (c^2 - v1^2) tau^2 - 2 (X.v1) tau -
//     |X|^2 = 0, whose half-discriminant is Dh: tau = (X.v1 + sqrt(Dh)) / (c^2 - v1^2), or |X|^2 / (sqrt(Dh) -
//     X.v1) for X.v1 < 0. The sum never cancels, where eq:dt's quadratic about t1 loses (c (t_n - t1) / R)^2;
//   - on the light cone |eta| = c tau, so no root or division by R is left: with kappa = c R - eta.v =
//     sqrt(Dh) - (t_r - t1) eta.a, A = c^2 - v^2 + eta.a and H = A v + kappa a, eq:LW_E and eq:LW_B become
//       E = q c (A eta - tau H) / kappa^3,   c^2 B = q c (H x eta) / kappa^3;
//   - the parts that one source shares with every target (its oldest slot's line, v, c^2 - v^2 and weights)
//     come from ext64, formed once per step and source.
// Against the same inputs in 113 bits, pairs and sums are off by 0.3 to 0.9 of what the previous form was (quadratic
// about t1, cross products; 50 and 118 operations) over gamma 2 to 197, and by under 1 % of it where R is far
// below c (t_n - t_{n-1}). One step, before and after: 45.8 and 29.6 ms at N = 16381 (251 slots, closed-form guess),
// 4.64 and 2.96 ms at N = 4096 (512 slots, bisection); 27.6 and 2.23 with the short work items and the target order it
// has now. The FP64 pipe is 90 % busy while an SM has work.
// SHAPE: targets per block (kBlock = shape_block(SHAPE); shapes 3 and 4 run as shape 0)
template <int PROP, bool ADAPT, bool MID, bool DUMP, int SHAPE>
__global__ void __launch_bounds__(shape_block(SHAPE)) pair_fp64_kernel(PairArgs a) {
  constexpr int kBlock = shape_block(SHAPE);
  __shared__ int s_item;
  __shared__ double2 s_e[kTile * (kExt64 / 2)];  // ext64 of the tile's sources
  // FP32 records of the tile's sources: the bisection's (hi, lo) of the oldest slot and of slot n - 1; with the
  // guess the present (hi, 1/gamma^2) and (dbeta, gamma^2), then (hi, lo) of the oldest slot
  __shared__ float4 s_f[kTile][4];
  __shared__ double s_acc[6][kBlock];  // per-thread sums of E and B over the tiles
  const long long N = a.N;
  const int D = a.D;

  Window win;
  win.p0 = a.state->p0;
  win.D = D;
  win.nw = (int)(a.state->n - a.state->k0) + 1;
  win.err = a.err;
  const int nw = win.nw;
  const int pn = a.state->pn;
  const float inv_cdt = PROP != kPropBisect ? (float)(1.0 / (kC * a.state->dt)) : 0.f;
  const float invL = (float)(1.0 / (kC * a.state->dt * D));
  const int pprev = nw > 1 ? win.phys(nw - 2) : pn;  // slot n - 1 (or n)

  unsigned n_ooh = 0, n_sc = 0, n_bi = 0, n_tests = 0, n_fb = 0;
  double emin = __longlong_as_double(0x7ff0000000000000LL), vmax2 = 0.0;  // adaptive time step (Sec. 2.4)
  int errbits = 0;

  // persistent blocks pull (source chunk, target tile) items, chunk-major, until none is left
  if (threadIdx.x == 0) s_item = -1;
  for (;;) {
  __syncthreads();
  if (threadIdx.x == 0) s_item = next_item(s_item, a.nitems, a.work);
  __syncthreads();
  const int item = s_item;
  if (item >= a.nitems) break;
  int b, chunk_id, tb;
  decode_item(a.sched, a.nbunch, item, b, chunk_id, tb);
  const BunchDesc& bd = a.bunches[b];
  const BunchSched& bs = a.sched[b];
  const float3 bref = make_float3((float)bd.beta_ref[0], (float)bd.beta_ref[1], (float)bd.beta_ref[2]);
  const int boff = (int)bd.off, bend = boff + bd.n;
  const int i_loc = tb * kBlock + (int)threadIdx.x;
  const bool active = i_loc < bd.n;
  const int t_idx = boff + (active ? i_loc : 0);
  const int i = debug_index(a.order ? a.order[t_idx] : t_idx, boff, bend, a.err);

  const double* rr = a.rec64 + ((size_t)i * D + pn) * 6;
  const double r0 = rr[0], r1 = rr[1], r2 = rr[2];
  const double vi0 = ADAPT ? rr[3] : 0.0, vi1 = ADAPT ? rr[4] : 0.0, vi2 = ADAPT ? rr[5] : 0.0;  // v_i(t_n)
  // FP32 hi/lo split of the target's position: node tests run in FP32 against the guard-band thresholds
  // of the slot tables and fall back to the FP64 test between them (the decision is the FP64 one)
  const float* tq = a.rec32 + ((size_t)i * D + pn) * 12;
  const float rh0 = tq[0], rh1 = tq[1], rh2 = tq[2];
  const float rl0 = tq[4], rl1 = tq[5], rl2 = tq[6];
  const bool far_target = fmaxf(fabsf(rh0), fmaxf(fabsf(rh1), fabsf(rh2))) > 0.5f;
  // learned proposal: the mean position of the warp's targets, where the network is evaluated
  float3 rc = make_float3(0.f, 0.f, 0.f);
  if (PROP == kPropMlp) rc = mlp::warp_mean(active, rh0, rh1, rh2);
  float fac_lane = 1.f;  // delay factor of source j0 + lane of the current group of 32

  const int j_begin = boff + chunk_id * bs.chunk;
  const int j_end = min(bend, j_begin + bs.chunk);
#pragma unroll
  for (int c = 0; c < 6; c++) s_acc[c][threadIdx.x] = 0.0;

  for (int tile = j_begin; tile < j_end; tile += kTile) {
  const int tn = min(kTile, j_end - tile);
  __syncthreads();
  for (int q = threadIdx.x; q < tn * (kExt64 / 2); q += kBlock) s_e[q] = __ldg(a.ext64 + (size_t)tile * (kExt64 / 2) + q);
  for (int q = threadIdx.x; q < tn * 4; q += kBlock) {
    const int c = q & 3;
    const int js = debug_index(tile + (q >> 2), boff, bend, a.err);
    const int slot = PROP == kPropBisect ? (c < 2 ? win.p0 : pprev) : (c < 2 ? pn : win.p0);
    const int part = PROP == kPropBisect ? (c & 1) : (c == 1 ? 2 : (c & 1));
    s_f[q >> 2][c] = __ldg(reinterpret_cast<const float4*>(a.rec32) + ((size_t)js * D + slot) * 3 + part);
  }
  __syncthreads();
  FieldSums sum;  // over this tile's sources
  for (int jj = 0; (PROP == kPropMlp || active) && jj < tn; ++jj) {
    const int j = debug_index(tile + jj, boff, bend, a.err);  // tile + jj itself in a release build
    float fac = 1.f;
    if (PROP == kPropMlp) {
      // every 32 sources, the warp evaluates the network for the next 32 (one per lane) at its mean target
      // position; each pair then scales its uniform-motion delay by its source's factor
      const int l = jj & 31;
      if (l == 0) {
        __syncwarp();
        const int js = jj + (int)(threadIdx.x & 31);
        const bool v = js < tn;
        const int jr = v ? tile + js : j;
        const float4* qn = reinterpret_cast<const float4*>(a.rec32 + ((size_t)jr * D + pn) * 12);
        const float4 q0n = __ldg(qn), q2n = __ldg(qn + 2);
        const float4 q2p = __ldg(reinterpret_cast<const float4*>(a.rec32 + ((size_t)jr * D + pprev) * 12) + 2);
        fac_lane = mlp::warp_delay_factor(*a.net, v, rc.x - q0n.x, rc.y - q0n.y, rc.z - q0n.z, bref.x + q2n.x,
                                          bref.y + q2n.y, bref.z + q2n.z, q2n.x - q2p.x, q2n.y - q2p.y,
                                          q2n.z - q2p.z, invL, (float)D);
      }
      fac = __shfl_sync(0xffffffffu, fac_lane, l);
    }
    if (!active) continue;  // and stay in the loop for the next group's evaluation
    if (j == i) continue;
    const double* src = a.rec64 + (size_t)j * D * 6;
    const float4* src32 = reinterpret_cast<const float4*>(a.rec32 + (size_t)j * D * 12);
    // P(k) at physical slot p from its FP32 record: on the hi/lo split outside the guard band, else the FP64 test
    auto test32 = [&](float4 q0, float4 q1, int p) -> bool {
      const float d0 = (rh0 - q0.x) + (rl0 - q1.x), d1 = (rh1 - q0.y) + (rl1 - q1.y), d2 = (rh2 - q0.z) + (rl2 - q1.z);
      const float D2 = d0 * d0 + d1 * d1 + d2 * d2;
      const float4 tb = __ldg(a.tab32 + p);
      if (!far_target) {
        if (D2 > tb.x) return true;
        if (D2 < tb.x * kLowerRatio) return false;
      }
      n_fb += 1;
      return node_test(r0, r1, r2, src + p * 6, __ldg(a.lhs64 + p));
    };
    auto ntest = [&](int l) -> bool {
      const int p = win.phys(l);
      return test32(__ldg(src32 + 3 * p), __ldg(src32 + 3 * p + 1), p);
    };
    // ---- 1. bracket: offset l1 of the older node --------------------------------------------
    int l1, br;
    n_tests += 1;
    if (nw == 1) {
      // only the present slot exists: every pair is out of history
      l1 = 0;
      br = 0;
    } else if (PROP == kPropBisect) {
      if (test32(s_f[jj][0], s_f[jj][1], win.p0)) {
        l1 = 0;
        br = 0;
      } else {
        n_tests += 1;
        if (!test32(s_f[jj][2], s_f[jj][3], pprev)) {
          l1 = nw - 2;
          br = 1;
        } else {
          int lo = 0, hi = nw - 1;
          while (hi - lo > 1) {
            const int m = (lo + hi) >> 1;
            n_tests += 1;
            if (ntest(m))
              hi = m;
            else
              lo = m;
          }
          l1 = lo;
          br = 2;
        }
      }
    } else {
      // guarded galloping search from the uniform-motion delay (scaled by the network's factor with the learned
      // proposal)
      const int lg = uniform_motion_guess(rh0, rh1, rh2, s_f[jj][0], s_f[jj][1], bref,
                                          PROP == kPropMlp ? inv_cdt * fac : inv_cdt, nw);
      int lo, hi;
      bool ooh = false;
      if (lg == 0 ? test32(s_f[jj][2], s_f[jj][3], win.p0) : ntest(lg)) {
        hi = lg;
        int s = 1;
        for (;;) {
          if (hi == 0) {
            ooh = true;
            break;
          }
          lo = max(hi - s, 0);
          n_tests += 1;
          if (!ntest(lo)) break;
          hi = lo;
          s <<= 1;
        }
      } else {
        lo = lg;
        int s = 1;
        for (;;) {
          hi = lo + s;
          if (hi >= nw - 1) {
            hi = nw - 1;
            break;
          }
          n_tests += 1;
          if (ntest(hi)) break;
          lo = hi;
          s <<= 1;
        }
      }
      if (ooh) {
        l1 = 0;
        br = 0;
      } else {
        while (hi - lo > 1) {
          const int m = (lo + hi) >> 1;
          n_tests += 1;
          if (ntest(m))
            hi = m;
          else
            lo = m;
        }
        l1 = lo;
        br = (l1 == nw - 2) ? 1 : 2;
      }
    }
    if (br == 0)
      n_ooh++;
    else if (br == 1)
      n_sc++;
    else
      n_bi++;
    if (DUMP) a.dump[(size_t)i * N + j] = 4 * l1 + br;

    // ---- 2. the source's line at t_n ----------------------------------------------------------
    const double2* se = s_e + jj * (kExt64 / 2);
    const double cw = se[5].x;  // c w_j: the charge constant -e / (4 pi eps0) is applied once per target
    Line ln;
    double2 y01, y23, y45, ts;  // newer record, (t_n - t1, 1 / (t2 - t1))
    double w10, w11, w12;       // older position (eq:mid)
    if (br == 0) {
      // out of history (eq:linear2): the line through the oldest slot
      const double2 e0 = se[0], e1 = se[1], e2 = se[2], e3 = se[3], e4 = se[4];
      ln.X0 = (r0 - e0.x) - e1.y;
      ln.X1 = (r1 - e0.y) - e2.x;
      ln.X2 = (r2 - e1.x) - e2.y;
      ln.v0 = e3.x;
      ln.v1 = e3.y;
      ln.v2 = e4.x;
      ln.C2 = e4.y;
    } else {
      const int p1 = win.phys(l1);
      const int p2 = p1 + 1 == D ? 0 : p1 + 1;
      const double2* R1 = reinterpret_cast<const double2*>(src + p1 * 6);
      const double2* R2 = reinterpret_cast<const double2*>(src + p2 * 6);
      const double2 x01 = __ldg(R1), x23 = __ldg(R1 + 1), x45 = __ldg(R1 + 2);
      if (MID) y01 = __ldg(R2);
      y23 = __ldg(R2 + 1);
      y45 = __ldg(R2 + 2);
      ts = __ldg(a.tab64 + p1);
      w10 = x01.x;
      w11 = x01.y;
      w12 = x23.x;
      ln.v0 = x23.y;
      ln.v1 = x45.x;
      ln.v2 = x45.y;
      ln.X0 = fma(-ln.v0, ts.x, r0 - w10);
      ln.X1 = fma(-ln.v1, ts.x, r1 - w11);
      ln.X2 = fma(-ln.v2, ts.x, r2 - w12);
      ln.set_c2();
    }
    if (MID && br != 0) {
      // eq:mid: the midpoint of the bracket stands for the retarded time; eq:LW_E and eq:LW_B as they stand
      const double idt = ts.y;
      const double v0 = 0.5 * (ln.v0 + y23.y), v1 = 0.5 * (ln.v1 + y45.x), v2 = 0.5 * (ln.v2 + y45.y);
      const double a0 = (y23.y - ln.v0) * idt, a1 = (y45.x - ln.v1) * idt, a2 = (y45.y - ln.v2) * idt;
      const double e0 = r0 - 0.5 * (w10 + y01.x), e1 = r1 - 0.5 * (w11 + y01.y), e2 = r2 - 0.5 * (w12 + y23.x);
      const double R2s = e0 * e0 + e1 * e1 + e2 * e2;
      const double invR = rsqrt(R2s);
      const double R = R2s * invR;
      const double cinvR = kC * invR;
      const double vp0 = e0 * cinvR - v0, vp1 = e1 * cinvR - v1, vp2 = e2 * cinvR - v2;
      const double evp = e0 * vp0 + e1 * vp1 + e2 * vp2;
      if (!(R2s > 0.0) || !(evp > 0.0)) {
        errbits |= kErrCoincide;
        continue;
      }
      const double c2mv2 = kC * kC - (v0 * v0 + v1 * v1 + v2 * v2);
      // eta x (v' x a)
      const double xa0 = vp1 * a2 - vp2 * a1, xa1 = vp2 * a0 - vp0 * a2, xa2 = vp0 * a1 - vp1 * a0;
      const double ac0 = e1 * xa2 - e2 * xa1, ac1 = e2 * xa0 - e0 * xa2, ac2 = e0 * xa1 - e1 * xa0;
      const double ievp = recip_refined(evp);
      const double pref = (cw * (1.0 / kC) * R) * (ievp * ievp * ievp);
      const double E0 = pref * (c2mv2 * vp0 + ac0), E1 = pref * (c2mv2 * vp1 + ac1), E2 = pref * (c2mv2 * vp2 + ac2);
      sum.E[0] += E0;
      sum.E[1] += E1;
      sum.E[2] += E2;
      sum.B[0] += (e1 * E2 - e2 * E1) * cinvR;
      sum.B[1] += (e2 * E0 - e0 * E2) * cinvR;
      sum.B[2] += (e0 * E1 - e1 * E0) * cinvR;
      continue;
    }
    const double XX = ln.XX(), Xv = ln.Xv();
    const double Dh = fma(Xv, Xv, XX * ln.C2);  // c^2 [|X|^2 (1 - beta1^2) + (X.beta1)^2]
    if (!(positive_normal(ln.C2) && positive_normal(Dh))) {
      errbits |= (!positive_normal(ln.C2) || (br != 0 && Dh != Dh)) ? kErrDisc : kErrCoincide;
      continue;
    }
    // ---- 3. fields, and the adaptive step's interaction scale |eta_ij| = c tau, |v_i(t_n) - v_j(t_r)| ------
    const Root root(Dh);
    Retarded ret{0.0, ln.v0, ln.v1, ln.v2};
    if (br == 0) {
      if (ADAPT) ret.tau = line_delay(ln, XX, Xv, root.sqrt());
      heaviside_fields(ln, se[5].y, root, sum);
    } else if (!bracket_fields(ln, XX, Xv, root, ts.x, ts.y, y23.y, y45.x, y45.y, cw, sum, ret)) {
      errbits |= kErrCoincide;
      continue;
    }
    if (ADAPT) {
      const double R = kC * ret.tau;
      if (R >= a.eta_allow) {
        emin = fmin(emin, R);
        const double dv0 = vi0 - ret.v0, dv1 = vi1 - ret.v1, dv2 = vi2 - ret.v2;
        vmax2 = fmax(vmax2, dv0 * dv0 + dv1 * dv1 + dv2 * dv2);
      }
    }
  }  // sources of the tile
#pragma unroll
  for (int c = 0; c < 3; c++) {
    s_acc[c][threadIdx.x] += sum.E[c];
    s_acc[3 + c][threadIdx.x] += sum.B[c];
  }
  }  // tiles
  if (active) {
    double Et[3], Bt[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
      Et[c] = s_acc[c][threadIdx.x] * kFieldScale;
      Bt[c] = s_acc[3 + c][threadIdx.x] * (kFieldScale / (kC * kC));
    }
    if (bs.nchunk == 1) {
      for (int c = 0; c < 3; c++) {
        a.E[3 * i + c] = Et[c];
        a.B[3 * i + c] = Bt[c];
      }
    } else {
      double* o = a.out + ((size_t)chunk_id * N + i) * 6;
      for (int c = 0; c < 3; c++) {
        o[c] = Et[c];
        o[3 + c] = Bt[c];
      }
    }
  }
  if (ADAPT) {
    // this item's interaction scale into its bunch's slots (every lane of the warp takes part)
    reduce_scale(a.scale + 2 * b, emin, vmax2);
    emin = __longlong_as_double(0x7ff0000000000000LL);
    vmax2 = 0.0;
  }
  }  // work items
  // counters: one atomic per warp and counter
  n_ooh = __reduce_add_sync(0xffffffffu, n_ooh);
  n_sc = __reduce_add_sync(0xffffffffu, n_sc);
  n_bi = __reduce_add_sync(0xffffffffu, n_bi);
  n_tests = __reduce_add_sync(0xffffffffu, n_tests);
  n_fb = __reduce_add_sync(0xffffffffu, n_fb);
  errbits = __reduce_or_sync(0xffffffffu, errbits);
  if ((threadIdx.x & 31) == 0) {
    if (n_ooh) atomicAdd(a.stats + kStatOOH, (unsigned long long)n_ooh);
    if (n_sc) atomicAdd(a.stats + kStatShortcut, (unsigned long long)n_sc);
    if (n_bi) atomicAdd(a.stats + kStatBisect, (unsigned long long)n_bi);
    if (n_tests) atomicAdd(a.stats + kStatNodeTests, (unsigned long long)n_tests);
    if (n_fb) atomicAdd(a.stats + kStatGuard, (unsigned long long)n_fb);
    if (errbits) atomicOr(a.err, errbits);
  }
}

__global__ void zero_kernel(double* __restrict__ a, double* __restrict__ b, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    a[i] = 0.0;
    b[i] = 0.0;
  }
}

template <bool ADAPT, bool MID, int SHAPE>
int max_blocks_fp64(int proposal) {
  int nb = 0;
  constexpr int B = shape_block(SHAPE);
  if (proposal == kPropClosedForm)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_fp64_kernel<kPropClosedForm, ADAPT, MID, false, SHAPE>, B, 0);
  else if (proposal == kPropMlp)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_fp64_kernel<kPropMlp, ADAPT, MID, false, SHAPE>, B, 0);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, pair_fp64_kernel<kPropBisect, ADAPT, MID, false, SHAPE>, B, 0);
  return nb > 0 ? nb : 1;
}

// the adaptive-step and eq:mid instances and the bracket dump run the default shape only
int max_blocks_pair_fp64(int proposal, int variant, int shape) {
  if (variant == 2) return max_blocks_fp64<false, true, 0>(proposal);
  if (variant == 1) return max_blocks_fp64<true, false, 0>(proposal);
  if (shape == 1) return max_blocks_fp64<false, false, 1>(proposal);
  if (shape == 2) return max_blocks_fp64<false, false, 2>(proposal);
  return max_blocks_fp64<false, false, 0>(proposal);
}

template <bool ADAPT, bool MID, bool DUMP, int SHAPE>
void launch_fp64(int proposal, const PairLaunch& pl, const PairArgs& a, cudaStream_t st) {
  constexpr int B = shape_block(SHAPE);
  if (proposal == kPropClosedForm)
    pair_fp64_kernel<kPropClosedForm, ADAPT, MID, DUMP, SHAPE><<<pl.grid, B, 0, st>>>(a);
  else if (proposal == kPropMlp)
    pair_fp64_kernel<kPropMlp, ADAPT, MID, DUMP, SHAPE><<<pl.grid, B, 0, st>>>(a);
  else
    pair_fp64_kernel<kPropBisect, ADAPT, MID, DUMP, SHAPE><<<pl.grid, B, 0, st>>>(a);
}

cudaError_t launch_pair_fp64(const DeviceState& s, const int* order, int proposal, int reconstruction,
                             const AdaptParams& ap, const PairLaunch& pl, cudaStream_t st, int* dump) {
  PairArgs a;
  a.rec64 = s.rec64;
  a.rec32 = s.rec32;
  a.lhs64 = s.tab.lhs64;
  a.tab32 = s.tab.tab32;
  a.tab64 = s.tab.tab64;
  a.ext64 = s.ext64;
  a.state = s.state;
  a.out = s.partial;
  a.E = s.Eself;
  a.B = s.Bself;
  a.stats = s.stats;
  a.err = s.err;
  a.N = s.N;
  a.D = s.D;
  a.nbunch = s.nbunch;
  a.bunches = s.bunches;
  a.sched = s.sched;
  a.nitems = pl.nitems;
  a.work = s.work;
  a.net = s.mlp_image ? mlp::infer_image(s.mlp_image) : nullptr;
  a.scale = s.scale;
  a.eta_allow = ap.eta_allow;
  a.order = order;
  a.dump = dump;
  // the work counter is zeroed by the set-up launch or the post-pair launch before
  // the midpoint reconstruction runs with a fixed time step only (the host refuses the combination);
  // the bracket dump runs the method's instance (the brackets depend on neither variant)
  if (dump)
    launch_fp64<false, false, true, 0>(proposal, pl, a, st);
  else if (reconstruction == 1)
    launch_fp64<false, true, false, 0>(proposal, pl, a, st);
  else if (ap.on)
    launch_fp64<true, false, false, 0>(proposal, pl, a, st);
  else if (pl.shape == 1)
    launch_fp64<false, false, false, 1>(proposal, pl, a, st);
  else if (pl.shape == 2)
    launch_fp64<false, false, false, 2>(proposal, pl, a, st);
  else
    launch_fp64<false, false, false, 0>(proposal, pl, a, st);
  return cudaGetLastError();
}

cudaError_t launch_zero_self(const DeviceState& s, cudaStream_t st) {
  zero_kernel<<<(unsigned)((3 * s.N + 255) / 256), 256, 0, st>>>(s.Eself, s.Bself, 3 * s.N);
  return cudaGetLastError();
}

namespace {
__global__ void recip_probe_kernel(const double* __restrict__ x, double* __restrict__ y, long long n) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) y[k] = recip_refined(x[k]);
}
}  // namespace

void set_error_text(const char* msg);

}  // namespace emppp

extern "C" EMPPP_API emppp_status emppp_reciprocal_probe(const double* x, double* y, int64_t n, void* cuda_stream) {
  if (n < 0 || (n > 0 && (!x || !y))) {
    emppp::set_error_text("emppp_reciprocal_probe: n >= 0 and device arrays x, y are required");
    return EMPPP_ERR_ARG;
  }
  if (n == 0) return EMPPP_OK;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  emppp::recip_probe_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, y, (long long)n);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    emppp::set_error_text(cudaGetErrorString(e));
    return EMPPP_ERR_CUDA;
  }
  return EMPPP_OK;
}
