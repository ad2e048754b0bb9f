// Stage-1 -> stage-2 handoff and stage-2 transport (Sec. 2.7): after the switch the pair interaction is
// turned off (E = 0, B = B_geo) and the particles are advanced with a larger step in the background
// field alone. Particles are then independent: the transport kernel keeps each particle in registers
// for many steps, with the stage-1 push (push_math.cuh) reduced to E = 0, and writes the final state back as the
// single present history slot.
#include "emppp_internal.cuh"
#include "fp64_roots.cuh"
#include "push_math.cuh"
#include "shadow.cuh"

namespace emppp {

namespace {

constexpr int kSumThreads = 256;

// per bunch: sum_i w_i x_i (3) and sum_i w_i over the present positions, in a fixed order
__global__ void __launch_bounds__(kSumThreads) bunch_sums_kernel(DeviceState s) {
  __shared__ double sh[4][kSumThreads];
  const BunchDesc bd = s.bunches[blockIdx.x];
  const int pn = (int)(s.state->n % s.D);
  double acc[4] = {0, 0, 0, 0};
  for (int k = threadIdx.x; k < bd.n; k += kSumThreads) {
    const long long i = bd.off + k;
    const double* r = s.rec64 + ((size_t)i * s.D + pn) * 6;
    const double w = s.wts[i];
    acc[0] += w * r[0];
    acc[1] += w * r[1];
    acc[2] += w * r[2];
    acc[3] += w;
  }
  for (int c = 0; c < 4; c++) sh[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int w = kSumThreads / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
      for (int c = 0; c < 4; c++) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int c = 0; c < 4; c++) s.bsum[4 * blockIdx.x + c] = sh[c][0];
}

// x += shift of the particle's bunch on the present slot; the history restarts at the present slot
__global__ void translate_kernel(DeviceState s, const double* __restrict__ shifts) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n = s.state->n;
  const int pn = (int)(n % s.D);
  if (i == 0) s.state->hist_start = n;
  if (i >= s.N) return;
  const int b = s.bunch_of[i];
  double* r = s.rec64 + ((size_t)i * s.D + pn) * 6;
  const double x0 = r[0] + shifts[3 * b], x1 = r[1] + shifts[3 * b + 1], x2 = r[2] + shifts[3 * b + 2];
  r[0] = x0;
  r[1] = x1;
  r[2] = x2;
  float4 q[3];
  const BunchDesc& bd = s.bunches[b];
  shadow_record(bd.origin, bd.beta_ref, x0, x1, x2, r[3], r[4], r[5], gamma2_of_u(s.u[3 * i], s.u[3 * i + 1], s.u[3 * i + 2]),
                q);
  float4* o = reinterpret_cast<float4*>(s.rec32 + ((size_t)i * s.D + pn) * 12);
  o[0] = q[0];
  o[1] = q[1];
  o[2] = q[2];
}

// One transport step (E = 0): the push of push_math.cuh in fewer FP64 operations. v = u / gamma and gm2 = gamma^2 come
// from the step before, which ends with them. With E = 0, u^- = u and the Higuera-Cary kick
// u+ = s [u + (u.t) t + u x t], u' = u+ + u+ x t is the rotation u' = u + 2 s (u + u x t) x t, s = 1 / (1 + t^2), t =
// tau / gamma+; 2 s t is formed from tau directly. h is folded into the background field (tau = h B).
template <int KIND>
__device__ __forceinline__ void transport_step(double x[3], double u[3], double v[3], double& gm2, double xh[3],
                                               const BextParams& bp, double hdt, const double tb[3]) {
#pragma unroll
  for (int c = 0; c < 3; c++) xh[c] = fma(hdt, v[c], x[c]);
  if (KIND == 0) {
#pragma unroll
    for (int c = 0; c < 3; c++) x[c] = fma(hdt, v[c], xh[c]);
    return;
  }
  double t0 = tb[0], t1 = tb[1], t2 = tb[2];  // tau of a uniform field
  if (KIND == 2) {
    // tau = K [3 z r / r^5 - e_z / r^3], K = h mu0 m0 / (4 pi) = tb[0]
    const double r0 = xh[0] - bp.center[0], r1 = xh[1] - bp.center[1], r2 = xh[2] - bp.center[2];
    const double ir = Root(fma(r2, r2, fma(r1, r1, r0 * r0))).rsqrt();
    const double i2 = ir * ir, k = tb[0] * (i2 * ir), b = (3.0 * k) * (r2 * i2);
    t0 = b * r0;
    t1 = b * r1;
    t2 = fma(b, r2, -k);
  }
  const double tau2 = fma(t2, t2, fma(t1, t1, t0 * t0));
  const double us = fma(u[2], t2, fma(u[1], t1, u[0] * t0)) * (1.0 / kC);
  const double sigma = gm2 - tau2;
  const double g2 = 0.5 * (sigma + Root(fma(sigma, sigma, 4.0 * fma(us, us, tau2))).sqrt());  // gamma+^2
  const double ig = Root(g2).rsqrt();
  const double k2 = ((2.0 * g2) * ig) * recip_refined(g2 + tau2);  // 2 s / gamma+
  const double a0 = t0 * ig, a1 = t1 * ig, a2 = t2 * ig;
  const double b0 = t0 * k2, b1 = t1 * k2, b2 = t2 * k2;
  const double w0 = fma(u[1], a2, fma(-u[2], a1, u[0])), w1 = fma(u[2], a0, fma(-u[0], a2, u[1])),
               w2 = fma(u[0], a1, fma(-u[1], a0, u[2]));
  u[0] = fma(w1, b2, fma(-w2, b1, u[0]));
  u[1] = fma(w2, b0, fma(-w0, b2, u[1]));
  u[2] = fma(w0, b1, fma(-w1, b0, u[2]));
  gm2 = fma(fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0])), 1.0 / (kC * kC), 1.0);
  const double igv = Root(gm2).rsqrt();
#pragma unroll
  for (int c = 0; c < 3; c++) {
    v[c] = u[c] * igv;
    x[c] = fma(hdt, v[c], xh[c]);
  }
}

// nsteps transport steps of every particle from the present slot n; the result is written as slot
// n + nsteps (state advanced by the host-side caller through the slot time stamp argument). What bounds it: the FP64
// pipe, 86 operations per particle-step in a dipole (about 140 with the shared push and the library's roots). One warp
// per block, so that the SMs' shares differ by little (N = 120001: 25 or 24 warps an SM; with blocks of four, 28 or
// 24). 512 steps of 120001 particles: 16.1 ms before, 10.1 ms now. The rotation adds small terms to u where s [u + ...]
// rounded u three times, always the same way: after 512 steps of a bunch of gamma 20 at 4 Earth radii u is 6e-16 (rms; at
// most 3.5e-15) of |u| from an extended-precision run, before 4.7e-14 (9.2e-14).
constexpr int kTransportThreads = 32;

template <int KIND>
__global__ void __launch_bounds__(kTransportThreads) transport_kernel(DeviceState s, BextParams bp, double dt,
                                                                      int nsteps, double t_end) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long n = s.state->n;
  const int pn = (int)(n % s.D);
  const int pe = (int)((n + nsteps) % s.D);
  if (i >= s.N) return;
  const double* rec = s.rec64 + ((size_t)i * s.D + pn) * 6;
  double x[3] = {rec[0], rec[1], rec[2]};
  double u[3] = {s.u[3 * i], s.u[3 * i + 1], s.u[3 * i + 2]};
  const double h = -kQe * dt / (2.0 * kMe), hdt = 0.5 * dt;
  const double tb[3] = {KIND == 2 ? h * (kMu0 / (4.0 * kPi)) * bp.m0 : h * bp.b[0], h * bp.b[1], h * bp.b[2]};
  double gm2 = fma(fma(u[2], u[2], fma(u[1], u[1], u[0] * u[0])), 1.0 / (kC * kC), 1.0);
  const double ig = Root(gm2).rsqrt();
  double v[3] = {u[0] * ig, u[1] * ig, u[2] * ig}, xh[3], B[3];
  for (int k = 0; k < nsteps; k++) transport_step<KIND>(x, u, v, gm2, xh, bp, hdt, tb);
  background_b(bp, xh[0], xh[1], xh[2], B);  // the last step's field
  if (!isfinite(x[0] + x[1] + x[2] + u[0] + u[1] + u[2])) atomicOr(s.err, kErrNonFinite);
  for (int c = 0; c < 3; c++) {
    s.u[3 * i + c] = u[c];
    s.Eself[3 * i + c] = 0.0;
    s.Bself[3 * i + c] = 0.0;
    s.Bout[3 * i + c] = B[c];
  }
  double* r = s.rec64 + ((size_t)i * s.D + pe) * 6;
  reinterpret_cast<double2*>(r)[0] = make_double2(x[0], x[1]);
  reinterpret_cast<double2*>(r)[1] = make_double2(x[2], v[0]);
  reinterpret_cast<double2*>(r)[2] = make_double2(v[1], v[2]);
  float4 q[3];
  const BunchDesc& bd = s.bunches[s.bunch_of[i]];
  shadow_record(bd.origin, bd.beta_ref, x[0], x[1], x[2], v[0], v[1], v[2], gamma2_of_u(u[0], u[1], u[2]), q);
  float4* o = reinterpret_cast<float4*>(s.rec32 + ((size_t)i * s.D + pe) * 12);
  o[0] = q[0];
  o[1] = q[1];
  o[2] = q[2];
  if (i == 0) s.slot_t[pe] = t_end;
}

__global__ void transport_advance_kernel(StepState* st, int nsteps, double t_end) {
  st->n += nsteps;
  st->t = t_end;
  st->hist_start = st->n;
}

}  // namespace

cudaError_t launch_bunch_sums(const DeviceState& s, cudaStream_t st) {
  bunch_sums_kernel<<<s.nbunch, kSumThreads, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_translate(const DeviceState& s, const double* shifts, cudaStream_t st) {
  translate_kernel<<<(unsigned)((s.N + 255) / 256), 256, 0, st>>>(s, shifts);
  return cudaGetLastError();
}

// nsteps transport steps ending at time t_end (accumulated by the caller one step at a time)
cudaError_t launch_transport_chunk(const DeviceState& s, const BextParams& b, double dt, int nsteps, double t_end,
                                   cudaStream_t st) {
  const unsigned blocks = (unsigned)((s.N + kTransportThreads - 1) / kTransportThreads);
  if (b.kind == 2)
    transport_kernel<2><<<blocks, kTransportThreads, 0, st>>>(s, b, dt, nsteps, t_end);
  else if (b.kind == 1)
    transport_kernel<1><<<blocks, kTransportThreads, 0, st>>>(s, b, dt, nsteps, t_end);
  else
    transport_kernel<0><<<blocks, kTransportThreads, 0, st>>>(s, b, dt, nsteps, t_end);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  transport_advance_kernel<<<1, 1, 0, st>>>(s.state, nsteps, t_end);
  return cudaGetLastError();
}

}  // namespace emppp
