// History ring (Sec. 2.2: positions and velocities stored at discrete steps; the acceleration is not
// stored) and per-step slot tables.
#include "emppp_internal.cuh"
#include "fp64_roots.cuh"
#include "setup.cuh"
#include "shadow.cuh"

namespace emppp {

// Writes record (j, p) of both rings from an FP64 position and velocity, gamma^2 and its inverse.
__device__ __forceinline__ void write_record(const DeviceState& s, long long j, int p, double w0, double w1, double w2,
                                             double v0, double v1, double v2, double gamma2, double inv_gamma2) {
  double* r = s.rec64 + ((size_t)j * s.D + p) * 6;
  reinterpret_cast<double2*>(r)[0] = make_double2(w0, w1);
  reinterpret_cast<double2*>(r)[1] = make_double2(w2, v0);
  reinterpret_cast<double2*>(r)[2] = make_double2(v1, v2);
  float4 q[3];
  const BunchDesc& bd = s.bunches[s.bunch_of[j]];
  shadow_record(bd.origin, bd.beta_ref, w0, w1, w2, v0, v1, v2, gamma2, inv_gamma2, q);
  float4* o = reinterpret_cast<float4*>(s.rec32 + ((size_t)j * s.D + p) * 12);
  o[0] = q[0];
  o[1] = q[1];
  o[2] = q[2];
}

__device__ __forceinline__ void write_record(const DeviceState& s, long long j, int p, double w0, double w1, double w2,
                                             double v0, double v1, double v2) {
  const double gamma2 = gamma2_of_v(v0, v1, v2);
  write_record(s, j, p, w0, w1, w2, v0, v1, v2, gamma2, 1.0 / gamma2);
}

// v = u / gamma with gamma = sqrt(1 + u.u / c^2), in the operation order of a plain FP64 evaluation
__device__ __forceinline__ void velocity_of(double u0, double u1, double u2, double& v0, double& v1, double& v2) {
  const double uu = __dadd_rn(__dadd_rn(__dmul_rn(u0, u0), __dmul_rn(u1, u1)), __dmul_rn(u2, u2));
  const double g = __dsqrt_rn(__dadd_rn(1.0, __ddiv_rn(uu, __dmul_rn(kC, kC))));
  v0 = __ddiv_rn(u0, g);
  v1 = __ddiv_rn(u1, g);
  v2 = __ddiv_rn(u2, g);
}

__global__ void init_slot0_kernel(DeviceState s, const double* __restrict__ x, const double* __restrict__ u,
                                  const double* __restrict__ w) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    s.slot_t[0] = 0.0;
    *s.err = 0;
  }
  if (i >= s.N) return;
  const double u0 = u[3 * i], u1 = u[3 * i + 1], u2 = u[3 * i + 2];
  double v0, v1, v2;
  velocity_of(u0, u1, u2, v0, v1, v2);
  write_record(s, i, 0, x[3 * i], x[3 * i + 1], x[3 * i + 2], v0, v1, v2);
  s.u[3 * i] = u0;
  s.u[3 * i + 1] = u1;
  s.u[3 * i + 2] = u2;
  s.wts[i] = w ? w[i] : 1.0;
  s.kq32[i] = (float)(-kQe * s.wts[i] / (4.0 * kPi * kEps0));
}

// slot p of every particle; dt > 0: the time since the slot before it, whose deviation (shadow.cuh) it completes
__global__ void scatter_slot_kernel(DeviceState s, int p, double dt, const double* __restrict__ W,
                                    const double* __restrict__ V) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= s.N) return;
  if (dt > 0.0) {
    const size_t q = (size_t)j * s.D + (p == 0 ? s.D - 1 : p - 1);
    const double* r = s.rec64 + q * 6;
    s.rec32[q * 12 + 7] =
        line_deviation(r[0], r[1], r[2], r[3], r[4], r[5], W[3 * j], W[3 * j + 1], W[3 * j + 2], dt);
  }
  write_record(s, j, p, W[3 * j], W[3 * j + 1], W[3 * j + 2], V[3 * j], V[3 * j + 1], V[3 * j + 2]);
}

// All slots of a history held on the device (W, V [nslots][N][3], the layout of emppp_set_history) in one launch:
// slot s goes to physical slot (p_first + s) mod D (last: these end with the present slot). What bounds it is memory, 24 +
// 24 bytes read and 96 written per record, and before that the stores: written by the thread that forms them, the
// 16-byte words of a record are half sectors, 32 lines to an instruction. So a block takes kScatterSlots consecutive
// slots of 32 particles, a record per thread, lays them out in shared memory as the rings have them and copies each
// particle's run out in one piece. N = 8192, 301 slots: 1.85 ms with one launch per slot, 0.25 with a thread's slots
// written in turn, 0.15 now, which FP64 work bounds (20 operations a record: 0.10; memory: 0.05).
constexpr int kScatterSlots = 8;
constexpr int kScatterRow = 3 * kScatterSlots + 1;  // float4s of a particle's run, and one that spreads the banks

__global__ void __launch_bounds__(32 * kScatterSlots) scatter_history_kernel(DeviceState s, int p_first, int nslots,
                                                                             int last, const double* __restrict__ W,
                                                                             const double* __restrict__ V) {
  __shared__ float4 s_rec[2][32][kScatterRow];  // FP64 and FP32 records
  const int lane = threadIdx.x & 31, slot = threadIdx.x >> 5;
  const long long j0 = (long long)blockIdx.x * 32, j = j0 + lane;
  const int k0 = blockIdx.y * kScatterSlots, k = k0 + slot;
  if (j < s.N && k < nslots) {
    const size_t at = ((size_t)k * s.N + j) * 3, next = at + (size_t)s.N * 3;
    const double w0 = __ldg(W + at), w1 = __ldg(W + at + 1), w2 = __ldg(W + at + 2);
    const double v0 = __ldg(V + at), v1 = __ldg(V + at + 1), v2 = __ldg(V + at + 2);
    double gamma2, ig2;
    record_gamma2(v0, v1, v2, gamma2, ig2);
    float4 q[3];
    const BunchDesc& bd = s.bunches[s.nbunch == 1 ? 0 : s.bunch_of[j]];
    shadow_record(bd.origin, bd.beta_ref, w0, w1, w2, v0, v1, v2, gamma2, ig2, q);
    if (!last || k + 1 < nslots) {  // the next slot, which may be another block's
      int p = (int)(((long long)p_first + k) % s.D);
      const double t = s.slot_t[p];
      p = p + 1 == s.D ? 0 : p + 1;
      q[1].w = line_deviation(w0, w1, w2, v0, v1, v2, __ldg(W + next), __ldg(W + next + 1), __ldg(W + next + 2),
                              s.slot_t[p] - t, ig2);
    }
    double2* r = reinterpret_cast<double2*>(&s_rec[0][lane][3 * slot]);
    r[0] = make_double2(w0, w1);
    r[1] = make_double2(w2, v0);
    r[2] = make_double2(v1, v2);
#pragma unroll
    for (int c = 0; c < 3; c++) s_rec[1][lane][3 * slot + c] = q[c];
  }
  __syncthreads();
  const int words = 3 * min(kScatterSlots, nslots - k0), p0 = (int)(((long long)p_first + k0) % s.D);
  for (int q = threadIdx.x; q < 32 * 3 * kScatterSlots; q += 32 * kScatterSlots) {
    const int row = q / (3 * kScatterSlots), c = q % (3 * kScatterSlots);
    if (c >= words || j0 + row >= s.N) continue;
    const int p = (p0 + c / 3) % s.D;
    const size_t to = ((size_t)(j0 + row) * s.D + p) * 3 + c % 3;
    reinterpret_cast<float4*>(s.rec64)[to] = s_rec[0][row][c];
    reinterpret_cast<float4*>(s.rec32)[to] = s_rec[1][row][c];
  }
}

__global__ void gather_slot_kernel(DeviceState s, int p, double* __restrict__ W, double* __restrict__ V) {
  const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= s.N) return;
  const double* r = s.rec64 + ((size_t)j * s.D + p) * 6;
  for (int c = 0; c < 3; c++) {
    if (W) W[3 * j + c] = r[c];
    if (V) V[3 * j + c] = r[3 + c];
  }
}

__global__ void set_state_kernel(DeviceState s, long long n, double t, double dt, long long hist_start,
                                 const double* __restrict__ u, const double* __restrict__ w) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    s.state->n = n;
    s.state->t = t;
    s.state->dt = dt;
    s.state->hist_start = hist_start;
    *s.err = 0;
  }
  if (i >= s.N) return;
  if (u) {
    s.u[3 * i] = u[3 * i];
    s.u[3 * i + 1] = u[3 * i + 1];
    s.u[3 * i + 2] = u[3 * i + 2];
  }
  s.wts[i] = w ? w[i] : 1.0;
  s.kq32[i] = (float)(-kQe * s.wts[i] / (4.0 * kPi * kEps0));
}

// Per-step slot tables over the usable window k0..n alone (used before the delay sampler).
__global__ void prep_kernel(DeviceState s) {
  const long long n = s.state->n;
  const double t_n = s.state->t;
  const long long hs = s.state->hist_start;
  const long long k0 = n - s.D + 1 > hs ? n - s.D + 1 : hs;
  const int p0 = (int)(k0 % s.D);
  const int pn = (int)(n % s.D);
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    s.state->k0 = k0;
    s.state->p0 = p0;
    s.state->pn = pn;
  }
  const int nwin = (int)(n - k0 + 1);
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < nwin; l += gridDim.x * blockDim.x) slot_table(s, l, p0, pn, nwin, t_n);
}

// Set-up of the pair kernel, for a step that the post-pair launch of the step before did not prepare: the window k0..n
// and its slot tables (as prep_kernel), the pair kernel's work counter, and, for the mixed path, per-source vectors
// (eq:linear at t_n):
//   P_j = w_{j,n-1} + v_{j,n-1} (t_n - t_{n-1}), the end of the last history segment, split hi/lo about
//     the bunch origin. For a pair in the near-field shortcut bracket [n-1, n] the retarded point is
//     written as P_j - v_{j,n-1} tau with tau = t_n - t_r: the same point as w_{j,n-1} + v_{j,n-1}
//     (t_r - t_{n-1}), with FP32 precision kept when c tau is far below c (t_n - t_{n-1}).
//   X_j = w_{j,k0} + v_{j,k0} (t_n - t_{k0}) - w_{j,n}, where the straight line of eq:linear2 (the
//     out-of-history case) is at t_n, relative to the source's present position. Along that line the
//     source moves uniformly, so its field is Heaviside's field about the point w_{j,n} + X_j; the
//     separation from a target is then (r - w_{j,n}) - X_j, formed without cancellation.
//   c_j = w_{j,n} - w_{j,k0} and T (1 + 32u) - |c_j|^2 (1 - 32u), rounded up, with T the FP32 upper
//     threshold of slot k0 (and at least 0, so that d = 0 never passes): the oldest-slot bound (kChordMargin),
//     by which an out-of-history pair's node test of slot k0 needs no record of that slot; and the FP32 record's beta - beta_ref,
//     1/gamma^2 and gamma^2 of slot k0, which Heaviside's field of that pair reads.
// For the FP64 path, per source, the out-of-history line of eq:linear2 in FP64 (kExt64): the present position,
// X_j of the same line, its velocity and the factors of Heaviside's field that no target changes.
__global__ void setup_kernel(DeviceState s, SetupExt extrap) {
  const long long n = s.state->n;
  const double t_n = s.state->t;
  const long long hs = s.state->hist_start;
  const long long k0 = n - s.D + 1 > hs ? n - s.D + 1 : hs;
  const int p0 = (int)(k0 % s.D);
  const int pn = (int)(n % s.D);
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid == 0) {
    s.state->k0 = k0;
    s.state->p0 = p0;
    s.state->pn = pn;
    *s.work = 0;
  }
  const int nwin = (int)(n - k0 + 1);
  if (gid < nwin) slot_table(s, (int)gid, p0, pn, nwin, t_n);
  if (extrap == SetupExt::none || gid >= s.N) return;
  const double* x = s.rec64 + ((size_t)gid * s.D + pn) * 6;
  const double T0 = t_n - s.slot_t[p0];
  Oldest o;
  o.load(s, extrap, gid, p0);
  if (extrap == SetupExt::fp64) {
    source_vectors_fp64(s, gid, x, o, T0);
    return;
  }
  const int p1 = pn == 0 ? s.D - 1 : pn - 1;
  source_vectors_mixed(s, gid, x, o, T0, n > k0 ? s.rec64 + ((size_t)gid * s.D + p1) * 6 : nullptr,
                       t_n - s.slot_t[p1]);
}

__global__ void reset_scale_kernel(DeviceState s) {
  for (int b = 0; b < s.nbunch; b++) {
    s.scale[2 * b] = (unsigned long long)0x7ff0000000000000ULL;
    s.scale[2 * b + 1] = 0ull;
  }
  s.adapt_info[0] = s.state->dt;
  s.adapt_info[1] = 0.0;
  s.adapt_info[2] = 0.0;
}

// results into arrays of the caller's, unless a device error is pending: the present positions to x, and [3N] from sa to
// da and sb to db (each destination may be null)
__global__ void deliver_kernel(DeviceState s, double* __restrict__ x, double* __restrict__ da, const double* __restrict__ sa,
                               double* __restrict__ db, const double* __restrict__ sb) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= 3 * s.N || *s.err != 0) return;
  if (x) x[q] = s.rec64[((size_t)(q / 3) * s.D + (size_t)(s.state->n % s.D)) * 6 + q % 3];
  if (da) da[q] = sa[q];
  if (db) db[q] = sb[q];
}

static inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

cudaError_t launch_init_slot0(const DeviceState& s, const double* x, const double* u, const double* w,
                              cudaStream_t st) {
  init_slot0_kernel<<<blocks_for(s.N, 256), 256, 0, st>>>(s, x, u, w);
  return cudaGetLastError();
}

cudaError_t launch_scatter_slot(const DeviceState& s, int p, double dt, const double* W, const double* V,
                                cudaStream_t st) {
  scatter_slot_kernel<<<blocks_for(s.N, 256), 256, 0, st>>>(s, p, dt, W, V);
  return cudaGetLastError();
}

cudaError_t launch_scatter_history(const DeviceState& s, int p_first, int nslots, const double* W, const double* V,
                                   cudaStream_t st) {
  // a single slot would leave seven of a block's eight warps idle (1e6 particles: 233 us, 167 this way)
  if (nslots == 1) return launch_scatter_slot(s, p_first, 0.0, W, V, st);
  // blockIdx.y counts groups of slots: at most 65535 of them per launch
  constexpr int kMost = 65535 * kScatterSlots;
  for (int k = 0; k < nslots; k += kMost) {
    const int m = nslots - k < kMost ? nslots - k : kMost;
    scatter_history_kernel<<<dim3(blocks_for(s.N, 32), blocks_for(m, kScatterSlots)), 32 * kScatterSlots, 0, st>>>(
        s, (int)(((long long)p_first + k) % s.D), m, k + m == nslots, W + (size_t)k * s.N * 3, V + (size_t)k * s.N * 3);
  }
  return cudaGetLastError();
}

cudaError_t launch_gather_slot(const DeviceState& s, int p, double* W, double* V, cudaStream_t st) {
  gather_slot_kernel<<<blocks_for(s.N, 256), 256, 0, st>>>(s, p, W, V);
  return cudaGetLastError();
}

cudaError_t launch_set_state(const DeviceState& s, long long n, double t, double dt, long long hist_start,
                             const double* u, const double* w, cudaStream_t st) {
  set_state_kernel<<<blocks_for(s.N, 256), 256, 0, st>>>(s, n, t, dt, hist_start, u, w);
  return cudaGetLastError();
}

cudaError_t launch_prep(const DeviceState& s, cudaStream_t st) {
  prep_kernel<<<1, 1024, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_setup(const DeviceState& s, SetupExt ext, cudaStream_t st) {
  const long long n = ext != SetupExt::none && s.N > s.D ? s.N : s.D;
  // small blocks: the per-slot and per-source FP64 work spreads over more SMs (an FP64 warp instruction
  // holds an SM's FP64 pipe for 16 cycles)
  setup_kernel<<<blocks_for(n, 64), 64, 0, st>>>(s, ext);
  return cudaGetLastError();
}

cudaError_t launch_reset_scale(const DeviceState& s, cudaStream_t st) {
  reset_scale_kernel<<<1, 1, 0, st>>>(s);
  return cudaGetLastError();
}

cudaError_t launch_deliver(const DeviceState& s, double* x, double* da, const double* sa, double* db, const double* sb,
                           cudaStream_t st) {
  deliver_kernel<<<blocks_for(3 * s.N, 256), 256, 0, st>>>(s, x, da, sa, db, sb);
  return cudaGetLastError();
}

}  // namespace emppp
