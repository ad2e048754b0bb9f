// Higuera-Cary push (Sec. 2.3, Ripperda form) with the background field (Sec. 2.6) and the append of
// the new history slot (Sec. 2.2).
//
// Per particle: x^{n+1/2} = x^n + (dt/2) v^n; B = B_self + B_ext(x^{n+1/2}); h = q dt / (2 m);
//   u^- = u^n + h E;  gamma^- = sqrt(1 + u^-.u^- / c^2);  tau = h B;  u* = u^-.tau / c;
//   sigma = gamma^-^2 - tau^2;  gamma^+ = sqrt((sigma + sqrt(sigma^2 + 4 (tau^2 + u*^2))) / 2);
//   t = tau / gamma^+;  s = 1 / (1 + t^2);  u^+ = s [u^- + (u^-.t) t + u^- x t];
//   u^{n+1} = u^+ + h E + u^+ x t   (u^+ x t, not the u^- x t misprint the paper warns about);
//   v^{n+1} = u^{n+1} / gamma^{n+1};  x^{n+1} = x^{n+1/2} + (dt/2) v^{n+1}.
// Then slot n+1 (modulo D) receives (x^{n+1}, v^{n+1}) and the time stamp t_n + dt.
// O(N) work; FP64 throughout (the momentum update needs it). The launch also sums the pair kernel's
// per-chunk partial fields, picks the adaptive step and advances the clock, so that a step after the
// pair kernel is one launch.
#include "emppp_internal.cuh"
#include "energy.cuh"
#include "fp64_roots.cuh"
#include "push_math.cuh"
#include "setup.cuh"
#include "shadow.cuh"

namespace emppp {

// Step size of the push from the pair kernel's per-bunch interaction scales (Sec. 2.4): each bunch's
// dt_b = c_dt eta_min,b / v_max,b clamped to [dt_min, dt_max] (dt_max when no pair qualified or v_max = 0);
// the step of all bunches (one clock) is the smallest dt_b. eta_rep and v_rep are the binding bunch's.
__device__ __forceinline__ double adaptive_step(const DeviceState& s, const AdaptParams& ap, double& eta_rep,
                                                double& v_rep) {
  double dt = ap.dt_max;
  eta_rep = 0.0;
  v_rep = 0.0;
  for (int b = 0; b < s.nbunch; b++) {
    const double eta_min = __longlong_as_double((long long)s.scale[2 * b]);
    const double v_max = sqrt(__longlong_as_double((long long)s.scale[2 * b + 1]));
    const bool bounded = v_max > 0.0 && eta_min < __longlong_as_double(0x7ff0000000000000LL);
    const double dtb = fmin(ap.dt_max, fmax(ap.dt_min, bounded ? ap.c_dt * eta_min / v_max : ap.dt_max));
    if (b == 0 || dtb < dt) {
      dt = dtb;
      eta_rep = bounded ? eta_min : 0.0;
      v_rep = v_max;
    }
  }
  return dt;
}

// Half-step field point (comparison variant, fixed dt): before the pair evaluation of step n every
// particle's history gains a provisional slot n+1 holding its half-drifted position
// x^{n+1/2} = x^n + (dt/2) v^n (the push's own half drift, same operations) and v^n, stamped t_n + dt/2,
// and the clock moves to (n+1, t_n + dt/2), so that the set-up and pair launches evaluate the fields
// there. The post-pair launch (half = 1) then pushes from slot n and overwrites slot n+1. The last block
// to finish moves the clock, as in the post-pair launch.
__global__ void half_slot_kernel(DeviceState s) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const StepState st = *s.state;
  const int pn = (int)(st.n % s.D);
  const int pnext = pn + 1 == s.D ? 0 : pn + 1;
  if (i == 0) s.slot_t[pnext] = st.t + 0.5 * st.dt;
  if (i < s.N) {
    const double* rec = s.rec64 + ((size_t)i * s.D + pn) * 6;
    const double u0 = s.u[3 * i], u1 = s.u[3 * i + 1], u2 = s.u[3 * i + 2];
    const double ig0 = rsqrt(1.0 + (u0 * u0 + u1 * u1 + u2 * u2) * (1.0 / (kC * kC)));
    const double hdt = 0.5 * st.dt;
    const double v0 = u0 * ig0, v1 = u1 * ig0, v2 = u2 * ig0;
    const double x0 = rec[0] + hdt * v0, x1 = rec[1] + hdt * v1, x2 = rec[2] + hdt * v2;
    double* r = s.rec64 + ((size_t)i * s.D + pnext) * 6;
    reinterpret_cast<double2*>(r)[0] = make_double2(x0, x1);
    reinterpret_cast<double2*>(r)[1] = make_double2(x2, v0);
    reinterpret_cast<double2*>(r)[2] = make_double2(v1, v2);
    float4 q[3];
    const BunchDesc& bd = s.bunches[s.bunch_of[i]];
    shadow_record(bd.origin, bd.beta_ref, x0, x1, x2, v0, v1, v2, gamma2_of_u(u0, u1, u2), q);
    float4* o = reinterpret_cast<float4*>(s.rec32 + ((size_t)i * s.D + pnext) * 12);
    o[0] = q[0];
    o[1] = q[1];
    o[2] = q[2];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(s.done, 1u);
    if (prev == gridDim.x - 1) {
      s.state->n = st.n + 1;
      s.state->t = st.t + 0.5 * st.dt;
      *s.done = 0u;
    }
  }
}

// ---- the sum of each target's per-chunk partial fields ----------------------------------------------------
// A block of kEnergyThreads threads takes P particles. The chunks fall in eight classes (c mod 8); kSumThreads threads
// each own one 16-byte word of a particle's six sums and some of the classes, so that the reads of neighbouring
// threads follow one another and a thread has several in flight; the classes are then added in order. The result is
// the same whatever P, so a bunch's sums do not depend on what else the solver holds.
// What bounds it: memory for large systems, one round of L2 latency for small ones. (A thread per particle, which read
// its chunks one after another, and a warp per particle, whose lanes read 48 bytes N * 48 apart, took 95 us at
// N = 65536 and 82 us at 16381, with the push; a step of the paper's 400 macroparticles went from 53 to 47 us.)
constexpr int kClasses = 8;
constexpr int kSumThreads = 192;

template <int P>
struct ChunkSums {
  static constexpr int kWords = 3 * P;                         // 16-byte words of the block's sums
  static constexpr int kGroups = kSumThreads / kWords;         // threads that share a word
  static constexpr int kPerThread = kClasses / kGroups;        // classes of a thread
  static_assert(kGroups * kWords == kSumThreads && kPerThread * kGroups == kClasses, "words and classes divide the threads");
  double2 part[kClasses][kWords];
  double2 sum[kWords];
  int chunks[P];  // chunks of the particle's bunch; at most 1: the pair kernel wrote its fields itself

  // fills sum, and the solver's Eself and Bself, for particles i0 .. i0 + P - 1 (whole block; ends with a barrier)
  __device__ __forceinline__ void run(const DeviceState& s, long long i0) {
    if (threadIdx.x < P) {
      const long long i = i0 + threadIdx.x;
      chunks[threadIdx.x] = i < s.N ? s.sched[s.nbunch == 1 ? 0 : s.bunch_of[i]].nchunk : 0;
    }
    __syncthreads();
    if (threadIdx.x < kSumThreads) {
      const int w = threadIdx.x % kWords, g = threadIdx.x / kWords;
      const int S = chunks[w / 3];
      const size_t stride = (size_t)s.N * 3;
      const double2* src = reinterpret_cast<const double2*>(s.partial) + i0 * 3 + w;
      double2 acc[kPerThread];
#pragma unroll
      for (int k = 0; k < kPerThread; k++) acc[k] = make_double2(0.0, 0.0);
      if (S > 1) {
#pragma unroll 4
        for (int c0 = g * kPerThread; c0 < S; c0 += kClasses) {
#pragma unroll
          for (int k = 0; k < kPerThread; k++) {
            if (c0 + k < S) {
              const double2 v = __ldcg(src + (size_t)(c0 + k) * stride);
              acc[k].x += v.x;
              acc[k].y += v.y;
            }
          }
        }
      }
#pragma unroll
      for (int k = 0; k < kPerThread; k++) part[g * kPerThread + k][w] = acc[k];
    }
    __syncthreads();
    if (threadIdx.x < kWords) {
      const int w = threadIdx.x;
      if (chunks[w / 3] > 1) {
        double2 t = part[0][w];
#pragma unroll
        for (int k = 1; k < kClasses; k++) {
          t.x += part[k][w].x;
          t.y += part[k][w].y;
        }
        sum[w] = t;
        // words: (E0, E1), (E2, B0), (B1, B2)
        const long long i = i0 + w / 3;
        const int c = w % 3;
        if (c == 0) {
          s.Eself[3 * i] = t.x;
          s.Eself[3 * i + 1] = t.y;
        } else if (c == 1) {
          s.Eself[3 * i + 2] = t.x;
          s.Bself[3 * i] = t.y;
        } else {
          s.Bself[3 * i + 1] = t.x;
          s.Bself[3 * i + 2] = t.y;
        }
      }
    }
    __syncthreads();
  }
};

// particles per block: few for small systems, whose push then spreads over more SMs (an FP64 warp instruction holds an
// SM's FP64 pipe for 16 cycles however few of its lanes are active), a full warp of pushers for large ones
int post_particles(long long n) { return n <= 2432 ? 8 : (n <= 4864 ? 16 : 32); }

long long post_table_threads(long long n) {
  const int p = post_particles(n);
  return (n + p - 1) / p * (kEnergyThreads - kSumThreads);
}

template <int P>
__global__ void __launch_bounds__(kEnergyThreads) reduce_partials_kernel(DeviceState s) {
  __shared__ ChunkSums<P> sums;
  sums.run(s, (long long)blockIdx.x * P);
}

cudaError_t launch_reduce_partials(const DeviceState& s, cudaStream_t st) {
  const int p = post_particles(s.N);
  const unsigned blocks = (unsigned)((s.N + p - 1) / p);
  if (p == 8)
    reduce_partials_kernel<8><<<blocks, kEnergyThreads, 0, st>>>(s);
  else if (p == 16)
    reduce_partials_kernel<16><<<blocks, kEnergyThreads, 0, st>>>(s);
  else
    reduce_partials_kernel<32><<<blocks, kEnergyThreads, 0, st>>>(s);
  return cudaGetLastError();
}

// The rest of a step after the pair kernel, in one launch: the sum of each target's per-chunk partial
// fields, the adaptive step size, the push of every particle and the append of slot
// n+1, then (by the last block to finish) the clock advance n -> n+1, t -> t + dt and the reset of the
// interaction-scale reduction. The last block is found with a counter that every block increments once
// after its work; nothing waits on it. With next it also forms what the pair kernel of the next step needs (setup.cuh),
// so that step goes without its set-up launch (6 us and a gap between launches, of 43 us a step with the paper's 400
// macroparticles): the slot tables need the step size alone and are formed by the warps that sum no chunks while others
// push, the source vectors by a warp whose loads are there by then. With half = 1 (half-step field point) the clock
// already stands at
// the provisional slot n+1: the push starts from slot n, the provisional slot is overwritten and the
// clock moves from t_n + dt/2 to t_n + dt (formed from t_n, as without the variant).
// With a full warp of pushers a block's phases (sums, push, records) use different units, so four blocks of 64 registers
// to an SM beat two of 104: 196 us and 121 at N = 65536.
// P = kEnergyThreads: a thread per particle that does all of its particle's work, for systems without partial sums that
// would take more than one round of the blocks of 32, most of whose threads have nothing to do then. Eight steps without
// pair fields, 32 particles a block and a thread each: N = 10000 154 us and 200; 20000 220 and 195; 65536 385 and 286;
// 1e6 4250 and 2470.
template <int P>
__global__ void __launch_bounds__(kEnergyThreads, P == 32 ? 4 : 1) step_post_kernel(DeviceState s, BextParams bp, AdaptParams ap,
                                                                   int chunked, int half, SetupExt next, int dev,
                                                                   EnergyParams ep, EnergyMon* __restrict__ mon) {
  constexpr bool kOwn = P == kEnergyThreads;
  __shared__ ChunkSums<kOwn ? 8 : P> sums;  // (not used, and left out, with a thread per particle)
  __shared__ double s_step[3];
  __shared__ double s_new[kOwn ? 1 : P][12];  // pushed particles: x, u, and the slot before, x and v
  const long long i0 = (long long)blockIdx.x * P;
  const StepState st = *s.state;
  // slot of x^n, the slot the push writes and t_n
  const int pfrom = half ? (st.pn == 0 ? s.D - 1 : st.pn - 1) : st.pn;
  const int pnext = half ? st.pn : (st.pn + 1 == s.D ? 0 : st.pn + 1);
  const double t_n = half ? s.slot_t[pfrom] : st.t;
  // the adaptive step size (FP64 root and division), by a warp that sums no chunks
  if (ap.on && threadIdx.x == kSumThreads) s_step[0] = adaptive_step(s, ap, s_step[1], s_step[2]);
  // the particle this thread pushes, its state loaded before the sums are there
  const long long i = i0 + threadIdx.x;
  const bool pusher = threadIdx.x < P && i < s.N;
  double x[3], u[3], vn[3];
  if (pusher) {
    const double* rec = s.rec64 + ((size_t)i * s.D + pfrom) * 6;
    for (int c = 0; c < 3; c++) {
      x[c] = rec[c];
      vn[c] = rec[3 + c];
      u[c] = s.u[3 * i + c];
    }
  }
  const int task = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long it = kOwn ? i : i0 + lane;
  // whether this thread does task k of particle it
  auto does = [&](int k) { return kOwn ? pusher : task == k && lane < P && it < s.N; };
  // the next step's window (fixed here: half and next exclude one another)
  const bool slides = st.n + 1 - s.D + 1 > st.k0;
  const long long k0_next = slides ? st.k0 + 1 : st.k0;
  const int p0_next = !slides ? st.p0 : (st.p0 + 1 == s.D ? 0 : st.p0 + 1);
  const bool sets_up = next != SetupExt::none && does(3);
  Oldest old;
  double t_old = 0.0;
  auto load_oldest = [&] {
    old.load(s, next, it, p0_next);
    t_old = s.slot_t[p0_next];
  };
  if (!kOwn && sets_up) load_oldest();
  if (!kOwn && chunked)
    sums.run(s, i0);
  else if (ap.on)
    __syncthreads();  // s_step
  const double dt = ap.on ? s_step[0] : st.dt;
  constexpr int kTableFirst = kOwn ? 0 : kSumThreads;
  if (next != SetupExt::none && (int)threadIdx.x >= kTableFirst) {
    constexpr int kTableThreads = kEnergyThreads - kTableFirst;
    const int nwin = (int)(st.n + 1 - k0_next) + 1;
    for (int l = blockIdx.x * kTableThreads + (int)threadIdx.x - kTableFirst; l < nwin; l += gridDim.x * kTableThreads)
      slot_table(s, l, p0_next, pnext, nwin, t_n + dt);
  }
  if (i == 0) {
    s.slot_t[pnext] = t_n + dt;
    if (ap.on) {
      s.adapt_info[0] = dt;
      s.adapt_info[1] = s_step[1];
      s.adapt_info[2] = s_step[2];
    }
  }
  double own[12];
  if (pusher) {
    double E[3], Bs[3];
    if (!kOwn && chunked && sums.chunks[threadIdx.x] > 1) {
      const double2 a = sums.sum[3 * threadIdx.x], b = sums.sum[3 * threadIdx.x + 1], c = sums.sum[3 * threadIdx.x + 2];
      E[0] = a.x;
      E[1] = a.y;
      E[2] = b.x;
      Bs[0] = b.y;
      Bs[1] = c.x;
      Bs[2] = c.y;
    } else {
      for (int c = 0; c < 3; c++) {
        E[c] = s.Eself[3 * i + c];
        Bs[c] = s.Bself[3 * i + c];
      }
    }
    double* out = kOwn ? own : s_new[threadIdx.x];
    for (int c = 0; c < 3; c++) {
      out[6 + c] = x[c];
      out[9 + c] = vn[c];
    }
    double v[3], B[3];
    push_particle(x, u, E, Bs, bp, dt, v, B);
    for (int c = 0; c < 3; c++) {
      out[c] = x[c];
      out[3 + c] = u[c];
      s.u[3 * i + c] = u[c];
      s.Bout[3 * i + c] = B[c];
    }
    if (!isfinite(x[0] + x[1] + x[2] + u[0] + u[1] + u[2])) atomicOr(s.err, kErrNonFinite);
    // append slot n+1 to the FP64 ring
    double* r = s.rec64 + ((size_t)i * s.D + pnext) * 6;
    reinterpret_cast<double2*>(r)[0] = make_double2(x[0], x[1]);
    reinterpret_cast<double2*>(r)[1] = make_double2(x[2], v[0]);
    reinterpret_cast<double2*>(r)[2] = make_double2(v[1], v[2]);
    vn[0] = v[0];
    vn[1] = v[1];
    vn[2] = v[2];
  }
  if (!kOwn) __syncthreads();
  // What follows from the pushed state, by a warp each: the FP32 record, the monitor's term, how far slot n + 1 lies from
  // slot n's line (dev: the newer-node bound of the mixed path; without it the record keeps +inf, which the bound takes
  // as unknown), and the next step's source vectors
  const double* o = kOwn ? own : s_new[lane];
  if (kOwn && sets_up) load_oldest();
  if (sets_up) {
    const double T0 = (t_n + dt) - t_old;
    if (next == SetupExt::fp64)
      source_vectors_fp64(s, it, o, old, T0);
    else
      source_vectors_mixed(s, it, o, old, T0, o + 6, (t_n + dt) - t_n);
  }
  if (does(0)) {
    const BunchDesc& bd = s.bunches[s.nbunch == 1 ? 0 : s.bunch_of[it]];
    // gamma^2 = 1 + u.u / c^2 and its inverse without divisions (both are rounded to FP32)
    const double gamma2 = 1.0 + (o[3] * o[3] + o[4] * o[4] + o[5] * o[5]) * (1.0 / (kC * kC));
    float4 q[3];
    shadow_record(bd.origin, bd.beta_ref, o[0], o[1], o[2], vn[0], vn[1], vn[2], gamma2, recip_refined(gamma2), q);
    float4* w = reinterpret_cast<float4*>(s.rec32 + ((size_t)it * s.D + pnext) * 12);
    w[0] = q[0];
    w[1] = q[1];
    w[2] = q[2];
  }
  if (ep.on && does(1)) s.ke[it] = kinetic_term(o[3], o[4], o[5], s.wts[it]);
  if (dev && does(2))
    s.rec32[((size_t)it * s.D + pfrom) * 12 + 7] =
        line_deviation(o[6], o[7], o[8], o[9], o[10], o[11], o[0], o[1], o[2], (t_n + dt) - t_n);
  // the last block to finish advances the clock and resets the reduction for the next step (and, with
  // ep.on, evaluates the energy monitor of every bunch on the pushed state)
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(s.done, 1u);
    s_last = (prev == gridDim.x - 1);
    if (s_last) {
      s.state->n = half ? st.n : st.n + 1;
      s.state->t = t_n + dt;
      s.state->dt = dt;
      if (next != SetupExt::none) {
        s.state->k0 = k0_next;
        s.state->p0 = p0_next;
        s.state->pn = pnext;
        *s.work = 0;
      }
      if (ap.on) {
        for (int b = 0; b < s.nbunch; b++) {
          s.scale[2 * b] = (unsigned long long)0x7ff0000000000000ULL;  // +inf
          s.scale[2 * b + 1] = 0ull;
        }
      }
      *s.done = 0u;
    }
  }
  __syncthreads();
  if (ep.on && s_last) {
    __threadfence();
    for (int b = 0; b < s.nbunch; b++)
      energy_block(s, ep, mon, 0, b, half ? st.n : st.n + 1, t_n + dt, s.ke);
  }
}

cudaError_t launch_step_post(const DeviceState& s, const BextParams& b, const AdaptParams& ap, bool chunked, bool half,
                             SetupExt next, bool dev, const EnergyParams* ep, EnergyMon* mon, int num_sms,
                             cudaStream_t st) {
  EnergyParams e{0, 1, 0.0};
  if (ep) e = *ep;  // the energy monitor in the last block (small systems)
  const int p = !chunked && s.N > 32LL * 4 * num_sms ? kEnergyThreads : post_particles(s.N);
  const unsigned blocks = (unsigned)((s.N + p - 1) / p);
  const int c = chunked ? 1 : 0, h = half ? 1 : 0, dv = dev ? 1 : 0;
  if (p == kEnergyThreads) {
    step_post_kernel<kEnergyThreads><<<blocks, kEnergyThreads, 0, st>>>(s, b, ap, c, h, next, dv, e, mon);
    return cudaGetLastError();
  }
  if (p == 8)
    step_post_kernel<8><<<blocks, kEnergyThreads, 0, st>>>(s, b, ap, c, h, next, dv, e, mon);
  else if (p == 16)
    step_post_kernel<16><<<blocks, kEnergyThreads, 0, st>>>(s, b, ap, c, h, next, dv, e, mon);
  else
    step_post_kernel<32><<<blocks, kEnergyThreads, 0, st>>>(s, b, ap, c, h, next, dv, e, mon);
  return cudaGetLastError();
}

cudaError_t launch_half_slot(const DeviceState& s, cudaStream_t st) {
  half_slot_kernel<<<(unsigned)((s.N + 255) / 256), 256, 0, st>>>(s);
  return cudaGetLastError();
}

}  // namespace emppp
