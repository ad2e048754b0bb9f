// emppp_fields_noalloc: the FP64 self-field evaluation for callers that cannot let this library
// allocate device memory.
//
// Some callers own every byte of device memory themselves -- a framework whose caching allocator
// holds the GPU's memory, a service that runs under a fixed device-memory budget, a latency-critical
// loop in which a cudaMalloc could stall or fail once memory is nearly full. They can hand this
// library their inputs and outputs, but not let it take more. This entry point therefore keeps all
// of its working memory (per-slot tables, the spatial target order and the per-slice partial field sums of
// the source-split kernel) in one fixed file-scope device array, g_scratch, of kScratchBytes bytes, which every GPU
// that loads the library holds until the process exits. It calls no cudaMalloc, cudaFree or other
// allocating routine.
//
// Because every call shares g_scratch, two calls whose work overlaps on the GPU (different streams,
// or different host threads) race and may corrupt each other's results; serialise them. Each call
// overwrites every scratch word it reads before reading it, so nothing is left to clear between
// calls. The device address of g_scratch is looked up with cudaGetSymbolAddress the first time the
// entry point runs on a device (with that device current); that first call should come before any
// stream capture on the device. The looked-up address is kept for the life of the process, so the
// entry point does not support cudaDeviceReset (or any other replacement of the device's primary
// context) between its calls.
//
// A numeric fault of a pair (|v| >= c in the history, coincident particles, non-finite input) is not
// reported through a status: the affected target's E and B come out NaN and the call returns EMPPP_OK.
//
// The evaluation is the FP64 path's, reading the caller's history in the slot-major layout of
// emppp_set_history: the same brackets (a guarded search from the uniform-motion guess, every node test in the
// reference operation order or decided by a margin far above its rounding) and the same field forms
// (fp64_fields.cuh), with the targets in the spatial order of order.cu.
#include <mutex>

#include "../../include/emppp.h"
#include "emppp_internal.cuh"
#include "fp64_fields.cuh"

namespace emppp {
void set_error_text(const char* msg);
}

using namespace emppp;

namespace {

constexpr size_t kScratchBytes = size_t(16) << 20;  // 16 MiB
constexpr int kMaxSlots = 4096;
constexpr long long kMaxTargets = 348160;
// scratch: node-test table, slot table, then the target order and its keys, then the partial sums
constexpr size_t kTabOffset = kMaxSlots * sizeof(double);
constexpr size_t kOrderOffset = kTabOffset + kMaxSlots * sizeof(double2);
constexpr int kBlock = 128;
constexpr long long kMinOrdered = 512;  // fewest targets that are put in spatial order, less one
constexpr int kTile = 64;  // sources staged in shared memory at a time, and the pairs of one partial sum

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

// (c (t_n - t_k))^2 in the reference operation order; t_n - t_k and 1 / (t_{k+1} - t_k), k = 0..nslots-1
__global__ void na_tables_kernel(const double* __restrict__ T, int nslots, double* __restrict__ lhs,
                                 double2* __restrict__ tab) {
  const double tn = T[nslots - 1];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < nslots; k += gridDim.x * blockDim.x) {
    const double dt = __dsub_rn(tn, T[k]);
    const double ct = __dmul_rn(kC, dt);
    lhs[k] = __dmul_rn(ct, ct);
    tab[k] = make_double2(dt, k + 1 < nslots ? 1.0 / (T[k + 1] - T[k]) : 0.0);
  }
}

// P(k) for d = r - w_k: lhs <= |d|^2. The high words (20 mantissa bits) decide unless they are within one of each
// other, a relative margin of at least 2^-21 against roundings of 2^-52; else the reference operation order. This
// takes six operations of the FP64 pipe with the three of d, where that order and a comparison take nine.
__device__ __forceinline__ bool na_node_test(double d0, double d1, double d2, double lhs) {
  const int hs = __double2hiint(fma(d2, d2, fma(d1, d1, d0 * d0))), hl = __double2hiint(lhs);
  if (hs > hl + 1) return true;
  if (hs < hl - 1) return false;
  return lhs <= __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d1, d1)), __dmul_rn(d2, d2));
}

// One thread per target; blockIdx.y selects a slice of sources. Slot k of particle j is at
// W[(k * n + j) * 3]; the present slot is nslots - 1 and every slot is usable (k0 = 0). order: targets in spatial
// order, so that a warp's pairs mostly take the same branch. What bounds it: the FP64 pipe (fp64_fields.cuh). The
// tile's sources are staged with the factors that no target changes and, in FP32, what the guess reads. With the
// paper's bisection, its node tests in FP64, the quadratic about the older node, divisions and square roots in place
// of the refined approximations and targets in index order, n = 4096 with 200 slots took 6.71 ms; now 2.54 ms.
__global__ void __launch_bounds__(kBlock)
    na_pair_kernel(const double* __restrict__ W, const double* __restrict__ V, const double* __restrict__ wts,
                   const int* __restrict__ order, long long n, int nslots, long long chunk,
                   const double* __restrict__ lhs, const double2* __restrict__ tab, double* __restrict__ part,
                   double* __restrict__ E, double* __restrict__ B) {
  // oldest slot: position (3), velocity (3), c^2 - v^2, c w
  __shared__ double s_old[8][kTile];
  // present record about the block's first target: (position, 1/gamma^2), (beta, gamma^2 / (c mean dt))
  __shared__ float4 s_now[2][kTile];
  const int kn = nslots - 1;
  const size_t sstride = (size_t)n * 3;  // doubles between consecutive slots of one particle
  const double* Wn = W + (size_t)kn * sstride;
  const double* Vn = V + (size_t)kn * sstride;
  const long long t0 = (long long)blockIdx.x * kBlock, it = t0 + threadIdx.x;
  const bool active = it < n;
  const long long i = order ? order[active ? it : t0] : (active ? it : t0);
  const double* ro = Wn + 3 * (size_t)(order ? order[t0] : t0);
  const double o0 = ro[0], o1 = ro[1], o2 = ro[2];
  const double* ri = Wn + 3 * (size_t)i;
  const double r0 = ri[0], r1 = ri[1], r2 = ri[2];
  const float rf0 = (float)(r0 - o0), rf1 = (float)(r1 - o1), rf2 = (float)(r2 - o2);
  const double T0 = tab[0].x, lhs0 = lhs[0];
  const float inv_cdt = kn > 0 ? (float)(kn / (kC * T0)) : 0.f;  // of the mean slot spacing
  const long long j0 = (long long)blockIdx.y * chunk;
  const long long j1 = min(n, j0 + chunk);
  double Et[3] = {0, 0, 0}, Bt[3] = {0, 0, 0};
  bool bad = false;
  for (long long tile = j0; tile < j1; tile += kTile) {
    const int tn = (int)min((long long)kTile, j1 - tile);
    __syncthreads();
    if (threadIdx.x < tn) {
      const long long j = tile + threadIdx.x;
      const double* w = W + 3 * (size_t)j;
      const double* v = V + 3 * (size_t)j;
      double C2 = kC * kC;
      for (int c = 2; c >= 0; c--) {
        s_old[c][threadIdx.x] = w[c];
        s_old[3 + c][threadIdx.x] = v[c];
        C2 = fma(-v[c], v[c], C2);
      }
      s_old[6][threadIdx.x] = C2;
      s_old[7][threadIdx.x] = kC * (wts ? wts[j] : 1.0);
      const double* wn = Wn + 3 * (size_t)j;
      const double* vn = Vn + 3 * (size_t)j;
      const double b0 = vn[0] * (1.0 / kC), b1 = vn[1] * (1.0 / kC), b2 = vn[2] * (1.0 / kC);
      const float ig2 = (float)(1.0 - (b0 * b0 + b1 * b1 + b2 * b2));
      s_now[0][threadIdx.x] = make_float4((float)(wn[0] - o0), (float)(wn[1] - o1), (float)(wn[2] - o2), ig2);
      s_now[1][threadIdx.x] = make_float4((float)b0, (float)b1, (float)b2, inv_cdt / ig2);
    }
    __syncthreads();
    FieldSums sum;
    for (int jj = 0; active && jj < tn; ++jj) {
      const long long j = tile + jj;
      if (j == i) continue;
      const double* wj = W + 3 * (size_t)j;
      // ---- bracket: offset of the older node; (d0, d1, d2) = r - w there ---------------------------------
      int k1 = 0;
      bool ooh = true;
      double d0, d1, d2, q0, q1, q2;
      auto test = [&](int k) -> bool {  // P(k); leaves r - w_k in q
        const double* w = wj + (size_t)k * sstride;
        q0 = r0 - __ldg(w);
        q1 = r1 - __ldg(w + 1);
        q2 = r2 - __ldg(w + 2);
        return na_node_test(q0, q1, q2, __ldg(lhs + k));
      };
      auto test0 = [&]() -> bool {  // P(0) from the staged oldest slot
        q0 = r0 - s_old[0][jj];
        q1 = r1 - s_old[1][jj];
        q2 = r2 - s_old[2][jj];
        return na_node_test(q0, q1, q2, lhs0);
      };
      auto keep = [&]() {
        d0 = q0;
        d1 = q1;
        d2 = q2;
      };
      if (kn == 0) {  // a single slot: every pair is out of history
        test0();
      } else {
        const float4 g = s_now[0][jj], h = s_now[1][jj];
        const float x0 = rf0 - g.x, x1 = rf1 - g.y, x2 = rf2 - g.z;
        const float xb = x0 * h.x + x1 * h.y + x2 * h.z;
        const float sc = (xb + sqrtf(fmaxf(xb * xb + g.w * (x0 * x0 + x1 * x1 + x2 * x2), 0.f))) * h.w;
        int lo, hi = max(kn - 1 - __float2int_rz(fmaxf(sc, 0.f)), 0), st = 1;
        if (hi == 0 ? test0() : test(hi)) {
          // gallop down (P true at hi)
          while (hi > 0) {
            lo = max(hi - st, 0);
            if (!(lo == 0 ? test0() : test(lo))) {
              keep();
              ooh = false;
              break;
            }
            hi = lo;
            st <<= 1;
          }
        } else {
          // gallop up (P false at lo; P(kn) is true)
          keep();
          ooh = false;
          lo = hi;
          for (;;) {
            hi = lo + st;
            if (hi >= kn) {
              hi = kn;
              break;
            }
            if (test(hi)) break;
            keep();
            lo = hi;
            st <<= 1;
          }
        }
        if (!ooh) {
          while (hi - lo > 1) {
            const int m = (lo + hi) >> 1;
            if (test(m)) {
              hi = m;
            } else {
              keep();
              lo = m;
            }
          }
          k1 = lo;
        }
      }
      // ---- the source's line at t_n, and the fields ------------------------------------------------------
      Line ln;
      double T1 = T0, idt = 0.0, u0, u1, u2;
      if (ooh) {
        keep();  // the last test was slot 0's
        ln.v0 = s_old[3][jj];
        ln.v1 = s_old[4][jj];
        ln.v2 = s_old[5][jj];
        ln.C2 = s_old[6][jj];
      } else {
        const double* v1 = V + 3 * (size_t)j + (size_t)k1 * sstride;
        const double* v2 = v1 + sstride;
        ln.v0 = __ldg(v1);
        ln.v1 = __ldg(v1 + 1);
        ln.v2 = __ldg(v1 + 2);
        u0 = __ldg(v2);
        u1 = __ldg(v2 + 1);
        u2 = __ldg(v2 + 2);
        const double2 ts = __ldg(tab + k1);
        T1 = ts.x;
        idt = ts.y;
        ln.set_c2();
      }
      ln.X0 = fma(-ln.v0, T1, d0);
      ln.X1 = fma(-ln.v1, T1, d1);
      ln.X2 = fma(-ln.v2, T1, d2);
      const double XX = ln.XX(), Xv = ln.Xv();
      const double Dh = fma(Xv, Xv, XX * ln.C2);
      if (!(positive_normal(ln.C2) && positive_normal(Dh))) {
        bad = true;
        continue;
      }
      const Root root(Dh);
      const double cw = s_old[7][jj];
      Retarded ret;
      if (ooh)
        heaviside_fields(ln, cw * ln.C2, root, sum);
      else if (!bracket_fields(ln, XX, Xv, root, T1, idt, u0, u1, u2, cw, sum, ret))
        bad = true;
    }
    for (int c = 0; c < 3; c++) {
      Et[c] += sum.E[c];
      Bt[c] += sum.B[c];
    }
  }
  if (!active) return;
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  for (int c = 0; c < 3; c++) {
    const double e = bad ? nan : Et[c] * kFieldScale, b = bad ? nan : Bt[c] * (kFieldScale / (kC * kC));
    if (part) {
      double* o = part + ((size_t)blockIdx.y * n + i) * 6;
      o[c] = e;
      o[3 + c] = b;
    } else {
      E[3 * i + c] = e;
      B[3 * i + c] = b;
    }
  }
}

// sum of the S slices' partial fields in slice order, a thread per component: the reads of a warp are contiguous
__global__ void na_reduce_kernel(const double* __restrict__ part, int S, long long n, double* __restrict__ E,
                                 double* __restrict__ B) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= 6 * n) return;
  double acc = 0.0;
#pragma unroll 8
  for (int s = 0; s < S; s++) acc += __ldg(part + (size_t)s * 6 * n + q);
  const long long i = q / 6;
  const int c = (int)(q - 6 * i);
  (c < 3 ? E + 3 * i + c : B + 3 * i + c - 3)[0] = acc;
}

// device address of g_scratch, looked up once per device
constexpr int kMaxDevices = 64;
std::mutex g_mu;
void* g_addr[kMaxDevices] = {};

emppp_status scratch_address(int dev, void** out) {
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) {
      set_error_text(cudaGetErrorString(e));
      return EMPPP_ERR_CUDA;
    }
    e = load_array_order();
    if (e != cudaSuccess) {
      set_error_text(cudaGetErrorString(e));
      return EMPPP_ERR_CUDA;
    }
    g_addr[dev] = p;
  }
  *out = g_addr[dev];
  return EMPPP_OK;
}

}  // namespace

extern "C" EMPPP_API emppp_status emppp_fields_noalloc(int64_t n, int32_t nslots, const double* T, const double* W,
                                                       const double* V, const double* w, double* E, double* B,
                                                       void* cuda_stream) {
  if (n < 1 || !T || !W || !V || !E || !B) {
    set_error_text("emppp_fields_noalloc: n >= 1 and non-NULL T, W, V, E, B are required");
    return EMPPP_ERR_ARG;
  }
  if (nslots < 1 || nslots > kMaxSlots) {
    set_error_text("emppp_fields_noalloc: nslots must be in 1..4096 (fixed scratch size)");
    return EMPPP_ERR_ARG;
  }
  if (n > kMaxTargets) {
    set_error_text("emppp_fields_noalloc: n exceeds the 16 MiB scratch limit (n <= 348160)");
    return EMPPP_ERR_ARG;
  }
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    set_error_text(e != cudaSuccess ? cudaGetErrorString(e) : "emppp_fields_noalloc: device index too large");
    return EMPPP_ERR_CUDA;
  }
  void* base = nullptr;
  emppp_status st = scratch_address(dev, &base);
  if (st != EMPPP_OK) return st;
  unsigned char* scratch = static_cast<unsigned char*>(base);
  double* lhs = reinterpret_cast<double*>(scratch);
  double2* tab = reinterpret_cast<double2*>(scratch + kTabOffset);
  int* order = reinterpret_cast<int*>(scratch + kOrderOffset);
  unsigned* key = reinterpret_cast<unsigned*>(order + n);
  const size_t part_offset = (kOrderOffset + (size_t)n * (sizeof(int) + sizeof(unsigned)) + 15) / 16 * 16;
  double* part = reinterpret_cast<double*>(scratch + part_offset);
  // Source slices: enough blocks for about sixteen per SM (their costs differ with their branch mix) if that leaves
  // slices of kLongSlice sources; a smaller system is bound by the chain of pairs in a thread and by what each
  // block sets up: about four blocks per SM, slices of kShortSlice sources at least (n = 100: 51 us, with slices of 32
  // 154; n = 600: 137 us, with eight blocks per SM 151). As far as the scratch holds their partial sums; a single slice writes
  // the fields itself.
  constexpr long long kLongSlice = 32, kShortSlice = 2;
  const long long ntb = (n + kBlock - 1) / kBlock;
  const long long fit = (long long)((kScratchBytes - part_offset) / ((size_t)n * 6 * sizeof(double)));
  long long S = (16LL * sms + ntb - 1) / ntb;
  if (S * kLongSlice > n) {
    S = (4LL * sms + ntb - 1) / ntb;
    if (S * kShortSlice > n) S = (n + kShortSlice - 1) / kShortSlice;
  }
  if (S > fit) S = fit;
  if (S < 1) S = 1;
  const long long chunk = (n + S - 1) / S;
  S = (n + chunk - 1) / chunk;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  na_tables_kernel<<<(nslots + 255) / 256, 256, 0, s>>>(T, nslots, lhs, tab);
  // the spatial order costs a launch (about 8 us), which a few target blocks do not repay (n = 300: 77 us without,
  // 87 with; n = 1000: 272 without, 266 with)
  const bool ordered = n > kMinOrdered;
  if (ordered) {
    e = launch_array_order(W + (size_t)(nslots - 1) * n * 3, V + (size_t)(nslots - 1) * n * 3, (int)n, key, order, s);
    if (e != cudaSuccess) {
      set_error_text(cudaGetErrorString(e));
      return EMPPP_ERR_CUDA;
    }
  }
  na_pair_kernel<<<dim3((unsigned)ntb, (unsigned)S), kBlock, 0, s>>>(W, V, w, ordered ? order : nullptr, n, nslots, chunk, lhs,
                                                                    tab,
                                                                    S > 1 ? part : nullptr, E, B);
  if (S > 1) na_reduce_kernel<<<(unsigned)((6 * n + 255) / 256), 256, 0, s>>>(part, (int)S, n, E, B);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error_text(cudaGetErrorString(e));
    return EMPPP_ERR_CUDA;
  }
  return EMPPP_OK;
}
