// Energy monitor of the stage switch (Sec. 2.7), one bunch per call by one block of threads: shared by
// the monitor's own launch and the last block of the post-pair launch, so that both compute the same
// values with the same operations.
#pragma once

#include "emppp_internal.cuh"

namespace emppp {

// kinetic-energy term of one particle, w (gamma - 1) / (m_e c^2) with gamma - 1 = (u.u / c^2) /
// (gamma + 1), in a fixed sequence of correctly rounded operations, so that the pushing thread and the
// monitor's own launch form the same value
__device__ __forceinline__ double kinetic_term(double u0, double u1, double u2, double w) {
  const double su = __fma_rn(u2, u2, __fma_rn(u1, u1, __dmul_rn(u0, u0)));
  const double uu = __ddiv_rn(su, kC * kC);
  return __dmul_rn(w, __ddiv_rn(uu, __dadd_rn(__dsqrt_rn(__dadd_rn(1.0, uu)), 1.0)));
}

// the monitor of bunch b, by one block of kEnergyThreads threads (also called by the last block of the
// post-pair launch, which has the same size); n, t: the present step and time. terms: the particles'
// kinetic_term values when already formed (by the pushing threads of the same launch), else nullptr.
// Reads of the particles go to L2 (__ldcg): they were written by other blocks of the same launch.
__device__ __forceinline__ void energy_block(const DeviceState& s, const EnergyParams& ep, EnergyMon* __restrict__ mon,
                                             int reset, int b, long long n, double t, const double* terms) {
  __shared__ double s_sum[2][kEnergyThreads];
  const BunchDesc& bd = s.bunches[b];
  EnergyMon m;
  if (threadIdx.x == 0) m = mon[b];
  double num = 0.0, den = 0.0;
  for (long long i = bd.off + threadIdx.x; i < bd.off + bd.n; i += kEnergyThreads) {
    const double w = __ldcg(s.wts + i);
    if (terms) {
      num += __ldcg(terms + i);
    } else {
      num += kinetic_term(__ldcg(s.u + 3 * i), __ldcg(s.u + 3 * i + 1), __ldcg(s.u + 3 * i + 2), w);
    }
    den += w;
  }
  // fixed tree, halving the distance: across the warps (by the first two warps, one sum each), then over their lanes
  s_sum[0][threadIdx.x] = num;
  s_sum[1][threadIdx.x] = den;
  __syncthreads();
  if (threadIdx.x < 64) {
    const int l = threadIdx.x & 31;
    const double* v = s_sum[threadIdx.x >> 5];
    static_assert(kEnergyThreads == 256, "the tree below adds eight warps");
    double t = ((v[l] + v[l + 128]) + (v[l + 64] + v[l + 192])) + ((v[l + 32] + v[l + 160]) + (v[l + 96] + v[l + 224]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (l == 0) s_sum[threadIdx.x >> 5][0] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    num = s_sum[0][0];
    den = s_sum[1][0];
    const double ebar = num / den * (kMe * kC * kC);
    if (reset) {
      m.ebar = ebar;
      m.rate = 0.0;
      m.t_prev = t;
      m.t_sw = 0.0;
      m.n_sw = -1;
      m.armed = 0;
      m.run = 0;
      m.switched = 0;
    } else {
      const double rate = (ebar - m.ebar) / (t - m.t_prev);
      m.rate = rate;
      m.ebar = ebar;
      m.t_prev = t;
      if (fabs(rate) >= ep.eps) m.armed = 1;
      m.run = (m.armed && fabs(rate) < ep.eps) ? m.run + 1 : 0;
      if (!m.switched && m.run >= ep.hold) {
        m.switched = 1;
        m.n_sw = n;
        m.t_sw = t;
      }
    }
    mon[b] = m;
  }
  __syncthreads();  // the shared arrays are reused for the next bunch
}

}  // namespace emppp
