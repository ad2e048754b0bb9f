// Spatial order of the targets for the pair kernels.
//
// Threads take targets in this order, so that the 32 targets of a warp are close in space: their retarded slots of any
// one source lie within a few cache lines, and they mostly take the same branch of the retarded-time search. Each
// bunch's present positions get a key along a Hilbert curve of 1024^3 cells; a counting sort lists the particles by the
// key's leading bits (6 to 15 from the bunch size), and windows of 2048 of the list are then sorted by the whole key.
// The delay of a source changes 1 + beta times as fast along the bunch's motion as across it, so that axis is
// stretched. (Branches that a warp takes for a source, N = 4096, 512 slots: 0.79 in history and 0.45 beyond with a
// Morton curve of the leading bits alone, 0.75 and 0.42 now; the FP64 step there 2.36 -> 2.22 ms, N = 16381 28.9 ->
// 27.6.) One block of 1024 threads sorts one bunch in shared memory: latency-bound, and rarely run. The order is a
// permutation of each bunch's index range (each target is evaluated exactly once whatever the order); the order inside
// a cell comes from shared-memory atomics and may differ run to run, which changes which thread evaluates a target but
// not its result.
#include "emppp_internal.cuh"

namespace emppp {

namespace {

constexpr int kThreads = 1024;
constexpr int kMaxBits = 5;
constexpr int kUnroll = 4;  // particles whose positions a thread loads before it uses any of them

constexpr int kKeyBits = 10;     // per axis
constexpr int kWindow = 2048;    // particles sorted by the whole key at a time

// index along the Hilbert curve of a cell (Skilling's transform of the axes, AIP Conf. Proc. 707, 381, 2004)
__device__ __forceinline__ unsigned hilbert_index(unsigned x, unsigned y, unsigned z) {
  for (unsigned q = 1u << (kKeyBits - 1); q > 1u; q >>= 1) {
    const unsigned p = q - 1u;
    if (x & q) x ^= p;
    auto fold = [&](unsigned& c) {
      if (c & q) {
        x ^= p;
      } else {
        const unsigned t = (x ^ c) & p;
        x ^= t;
        c ^= t;
      }
    };
    fold(y);
    fold(z);
  }
  y ^= x;
  z ^= y;
  unsigned t = 0;
  for (unsigned q = 1u << (kKeyBits - 1); q > 1u; q >>= 1)
    if (z & q) t ^= q - 1u;
  x ^= t;
  y ^= t;
  z ^= t;
  unsigned r = 0;
  for (int k = kKeyBits - 1; k >= 0; k--) r = (r << 3) | (((x >> k) & 1u) << 2) | (((y >> k) & 1u) << 1) | ((z >> k) & 1u);
  return r;
}

__host__ __device__ __forceinline__ int cell_bits(int n) {
  int lg = 0;
  while ((1 << (lg + 1)) <= n) lg++;
  int b = lg / 3;
  return b < 2 ? 2 : (b > kMaxBits ? kMaxBits : b);
}

// where the particles to order stand: the bunch of a block and the FP32 position of its particle k
struct RingPositions {  // present positions of a solver's bunches (hi parts about their origins)
  DeviceState s;
  const float4* rec;
  int pn;
  __device__ __forceinline__ void begin() {
    rec = reinterpret_cast<const float4*>(s.rec32);
    pn = (int)(s.state->n % s.D);
  }
  __device__ __forceinline__ int count() const { return s.bunches[blockIdx.x].n; }
  __device__ __forceinline__ long long offset() const { return s.bunches[blockIdx.x].off; }
  __device__ __forceinline__ float stretch(int c) const { return 1.f + fabsf((float)s.bunches[blockIdx.x].beta_ref[c]); }
  // one record per particle's ring run, so every particle is its own cache line
  __device__ __forceinline__ float4 at(long long k) const { return __ldg(rec + ((size_t)k * s.D + pn) * 3); }
};
struct ArrayPositions {  // x [n][3], about the first particle; v: its velocity
  const double* x;
  const double* v;
  int n;
  __device__ __forceinline__ void begin() {}
  __device__ __forceinline__ int count() const { return n; }
  __device__ __forceinline__ long long offset() const { return 0; }
  __device__ __forceinline__ float stretch(int c) const { return 1.f + fabsf((float)(__ldg(v + c) * (1.0 / kC))); }
  __device__ __forceinline__ float4 at(long long k) const {
    return make_float4((float)(__ldg(x + 3 * k) - __ldg(x)), (float)(__ldg(x + 3 * k + 1) - __ldg(x + 1)),
                       (float)(__ldg(x + 3 * k + 2) - __ldg(x + 2)), 0.f);
  }
};

template <class Positions>
__global__ void __launch_bounds__(kThreads) order_kernel(Positions where, unsigned* __restrict__ key,
                                                         int* __restrict__ order) {
  extern __shared__ __align__(16) int hist[];  // cell counts, then the window being sorted
  __shared__ float s_lo[3][32], s_hi[3][32];
  __shared__ int s_warp[32];
  where.begin();
  const int n = where.count();
  const long long off = where.offset();
  const int bits = cell_bits(n);
  const int cells = 1 << (3 * bits);
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

  // position of particle k of the bunch; kUnroll of them are loaded before any is used
  auto position = [&](int k) { return where.at(off + k); };
  // bounding box of the present FP32 positions
  float lo[3] = {3.0e38f, 3.0e38f, 3.0e38f}, hi[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
  for (int k0 = tid; k0 < n; k0 += kUnroll * kThreads) {
    float4 q[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
      const int k = k0 + u * kThreads;
      const float nan = __int_as_float(0x7fc00000);  // skipped by the box below
      q[u] = k < n ? position(k) : make_float4(nan, nan, nan, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
      const float x3[3] = {q[u].x, q[u].y, q[u].z};
      for (int c = 0; c < 3; c++) {
        const float x = x3[c];
        if (x == x) {
          lo[c] = fminf(lo[c], x);
          hi[c] = fmaxf(hi[c], x);
        }
      }
    }
  }
  for (int c = 0; c < 3; c++) {
    for (int o = 16; o > 0; o >>= 1) {
      lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
      hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
    }
    if (lane == 0) {
      s_lo[c][wid] = lo[c];
      s_hi[c][wid] = hi[c];
    }
  }
  for (int k = tid; k < cells; k += kThreads) hist[k] = 0;
  __syncthreads();
  // the box as a cube of stretched axes
  float blo[3], sc[3], side = 0.f;
  for (int c = 0; c < 3; c++) {
    float a = 3.0e38f, b2 = -3.0e38f;
    for (int w = 0; w < kThreads / 32; w++) {
      a = fminf(a, s_lo[c][w]);
      b2 = fmaxf(b2, s_hi[c][w]);
    }
    blo[c] = a;
    sc[c] = where.stretch(c);
    side = fmaxf(side, (b2 - a) * sc[c]);
  }
  const float to_cell = side > 0.f ? (float)(1 << kKeyBits) / side : 0.f;
  const int drop = 3 * (kKeyBits - bits);  // bits of the key that the counting sort leaves out
  // cell keys and histogram
  for (int k0 = tid; k0 < n; k0 += kUnroll * kThreads) {
    float4 q[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
      const int k = k0 + u * kThreads;
      q[u] = k < n ? position(k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; u++) {
      const int k = k0 + u * kThreads;
      if (k >= n) break;
      const float x3[3] = {q[u].x, q[u].y, q[u].z};
      unsigned cc[3];
      for (int c = 0; c < 3; c++) {
        float f = (x3[c] - blo[c]) * sc[c] * to_cell;
        f = (f == f) ? fminf(fmaxf(f, 0.f), (float)((1 << kKeyBits) - 1)) : 0.f;
        cc[c] = (unsigned)f;
      }
      const unsigned m = hilbert_index(cc[0], cc[1], cc[2]);
      key[off + k] = m;
      atomicAdd(hist + (m >> drop), 1);
    }
  }
  __syncthreads();
  // exclusive scan of the cell counts: each thread owns a contiguous run of cells
  const int per = (cells + kThreads - 1) / kThreads;
  const int c0 = tid * per, c1 = min(cells, c0 + per);
  int sum = 0;
  for (int k = c0; k < c1; k++) sum += hist[k];
  int x = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_warp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int w = s_warp[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    s_warp[lane] = w;
  }
  __syncthreads();
  int base = x - sum + (wid > 0 ? s_warp[wid - 1] : 0);
  for (int k = c0; k < c1; k++) {
    const int v = hist[k];
    hist[k] = base;
    base += v;
  }
  __syncthreads();
  // scatter
  for (int k = tid; k < n; k += kThreads) {
    const int pos = atomicAdd(hist + (key[off + k] >> drop), 1);
    order[off + pos] = (int)(off + k);
  }
  __syncthreads();
  // windows of the list by the whole key: bitonic sort of (key, particle), whose last strides stay inside a warp
  unsigned long long* win = reinterpret_cast<unsigned long long*>(hist);
  for (int w0 = 0; w0 < n; w0 += kWindow) {
    const int m = min(kWindow, n - w0);
    int size = 64;
    while (size < m) size <<= 1;
    for (int k = tid; k < size; k += kThreads) {
      const int p = k < m ? order[off + w0 + k] : 0;
      win[k] = k < m ? ((unsigned long long)key[p] << 32) | (unsigned)p : ~0ull;
    }
    __syncthreads();
    for (int len = 2; len <= size; len <<= 1) {
      for (int j = len >> 1; j > 0; j >>= 1) {
        if (tid < size / 2) {
          const int lo_k = 2 * tid - (tid & (j - 1));
          const unsigned long long u = win[lo_k], v = win[lo_k + j];
          if ((u > v) == ((lo_k & len) == 0)) {
            win[lo_k] = v;
            win[lo_k + j] = u;
          }
        }
        if (j > 32 || (j == 1 && len >= 64))
          __syncthreads();
        else
          __syncwarp();
      }
    }
    for (int k = tid; k < m; k += kThreads) order[off + w0 + k] = (int)(unsigned)win[k];
    __syncthreads();
  }
}

}  // namespace

constexpr size_t kSmem = sizeof(int) << (3 * kMaxBits);

// the largest bunch's cell counts or a window: a small system does not reserve 128 KB of shared memory
static size_t shared_bytes(int n) {
  const size_t cells = sizeof(int) << (3 * cell_bits(n)), window = sizeof(unsigned long long) * kWindow;
  return cells > window ? cells : window;
}

// allows the kernel its shared-memory histogram on the current device (call before launching)
cudaError_t prepare_target_order() {
  cudaError_t e =
      cudaFuncSetAttribute(order_kernel<RingPositions>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(order_kernel<ArrayPositions>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
}

cudaError_t launch_array_order(const double* x, const double* v, int n, unsigned* key, int* order, cudaStream_t st) {
  order_kernel<<<1, kThreads, shared_bytes(n), st>>>(ArrayPositions{x, v, n}, key, order);
  return cudaGetLastError();
}

cudaError_t launch_target_order(const DeviceState& s, unsigned* key, int* order, long long max_bunch, cudaStream_t st) {
  const size_t smem = shared_bytes((int)(max_bunch < (1LL << 30) ? max_bunch : (1LL << 30)));
  order_kernel<<<s.nbunch, kThreads, smem, st>>>(RingPositions{s, nullptr, 0}, key, order);
  return cudaGetLastError();
}

}  // namespace emppp
