// Spatial order of the targets for the pair kernels.
//
// Threads take targets in this order, so that the 32 targets of a warp are close in space: their retarded slots of any
// one source lie within a few cache lines, and they mostly take the same branch of the retarded-time search. Each
// bunch's present positions get a key along a Hilbert curve of 1024^3 cells; a counting sort lists the particles by the
// key's leading bits (6 to 15 from the bunch size), and windows of 2048 of the list are then sorted by the whole key.
// The delay of a source changes faster along the bunch's motion than across it, so that axis is stretched, by 1 + 2 beta
// (N = 6000 mixed: 451 us with 1 + beta, 441 with 1 + 2 beta; 4096 FP64 2268 and 2241). Branches that a warp takes for
// a source, N = 4096, 512 slots: 0.79 in history and 0.45 beyond with a Morton curve of the leading bits alone, 0.75 and
// 0.42 with 1 + beta; the FP64 step there 2.36 -> 2.24 ms, N = 16381 28.7 -> 27.6, the mixed step of 65536 29.0 -> 28.2.
// A bunch of more than 2048 particles is sorted by a cluster of eight blocks, each of which holds the counts of an
// eighth of the cells, a smaller one by one block: latency and the shared-memory sort bound it (N = 8192: 85 us with one
// block, 32 with eight; 65536: 697 and 100). The order is a permutation of each bunch's index range (each target is
// evaluated exactly once whatever the order); the order inside a cell comes from shared-memory atomics and may differ
// run to run, which changes which thread evaluates a target but not its result.
#include <cooperative_groups.h>

#include "emppp_internal.cuh"

namespace emppp {

namespace {

constexpr int kThreads = 1024;
constexpr int kMaxBits = 5;
constexpr int kUnroll = 4;  // particles whose positions a thread loads before it uses any of them

constexpr int kKeyBits = 10;     // per axis
constexpr int kWindow = 2048;    // particles sorted by the whole key at a time
constexpr int kCluster = 8;      // blocks of a bunch of more than kWindow particles
constexpr int kCells = 4096;     // cell counts of a block
static_assert((1 << (3 * kMaxBits)) <= kCluster * kCells && kCells * sizeof(int) == kWindow * sizeof(unsigned long long),
              "the cells of a bunch fit its blocks, and a window the place of a block's counts");

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
  int pn, bunch;
  __device__ __forceinline__ void begin(int b) {
    bunch = b;
    rec = reinterpret_cast<const float4*>(s.rec32);
    pn = (int)(s.state->n % s.D);
  }
  __device__ __forceinline__ int count() const { return s.bunches[bunch].n; }
  __device__ __forceinline__ long long offset() const { return s.bunches[bunch].off; }
  __device__ __forceinline__ float stretch(int c) const { return 1.f + 2.f * fabsf((float)s.bunches[bunch].beta_ref[c]); }
  // one record per particle's ring run, so every particle is its own cache line
  __device__ __forceinline__ float4 at(long long k) const { return __ldg(rec + ((size_t)k * s.D + pn) * 3); }
};
struct ArrayPositions {  // x [n][3], about the first particle; v: its velocity
  const double* x;
  const double* v;
  int n;
  __device__ __forceinline__ void begin(int) {}
  __device__ __forceinline__ int count() const { return n; }
  __device__ __forceinline__ long long offset() const { return 0; }
  __device__ __forceinline__ float stretch(int c) const { return 1.f + 2.f * fabsf((float)(__ldg(v + c) * (1.0 / kC))); }
  __device__ __forceinline__ float4 at(long long k) const {
    return make_float4((float)(__ldg(x + 3 * k) - __ldg(x)), (float)(__ldg(x + 3 * k + 1) - __ldg(x + 1)),
                       (float)(__ldg(x + 3 * k + 2) - __ldg(x + 2)), 0.f);
  }
};

template <class Positions>
__global__ void __launch_bounds__(kThreads) order_kernel(Positions where, unsigned* key, int* order) {
  __shared__ __align__(16) unsigned long long win[kWindow];  // the window being sorted; before that, cell counts
  int* hist = reinterpret_cast<int*>(win);
  __shared__ float s_lo[3][32], s_hi[3][32], s_box[6];
  __shared__ int s_warp[32], s_total;
  const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int rank = (int)cl.block_rank(), nblocks = (int)cl.num_blocks();
  where.begin((int)blockIdx.x / nblocks);
  const int n = where.count();
  const long long off = where.offset();
  const int bits = cell_bits(n);
  // this block's share of the particles' loops and of the cells
  const int step = nblocks * kUnroll * kThreads, begin = rank * kUnroll * kThreads;
  const int share = 3 * bits - (nblocks > 1 ? 3 : 0), cells = 1 << share;
  static_assert(kCluster == 8, "eight blocks take the key's first three bits");
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

  // position of particle k of the bunch; kUnroll of them are loaded before any is used
  auto position = [&](int k) { return where.at(off + k); };
  // bounding box of the present FP32 positions
  float lo[3] = {3.0e38f, 3.0e38f, 3.0e38f}, hi[3] = {-3.0e38f, -3.0e38f, -3.0e38f};
  for (int k0 = begin + tid; k0 < n; k0 += step) {
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
  if (tid < 3) {
    float a = 3.0e38f, b2 = -3.0e38f;
    for (int w = 0; w < kThreads / 32; w++) {
      a = fminf(a, s_lo[tid][w]);
      b2 = fmaxf(b2, s_hi[tid][w]);
    }
    s_box[tid] = a;
    s_box[3 + tid] = b2;
  }
  cl.sync();
  // the box as a cube of stretched axes
  float blo[3], sc[3], side = 0.f;
  for (int c = 0; c < 3; c++) {
    float a = 3.0e38f, b2 = -3.0e38f;
    for (int r = 0; r < nblocks; r++) {
      const float* box = cl.map_shared_rank(s_box, r);
      a = fminf(a, box[c]);
      b2 = fmaxf(b2, box[3 + c]);
    }
    blo[c] = a;
    sc[c] = where.stretch(c);
    side = fmaxf(side, (b2 - a) * sc[c]);
  }
  const float to_cell = side > 0.f ? (float)(1 << kKeyBits) / side : 0.f;
  const int drop = 3 * (kKeyBits - bits);  // bits of the key that the counting sort leaves out
  auto count_of = [&](unsigned m) { return cl.map_shared_rank(hist, (int)((m >> drop) >> share)) + ((m >> drop) & (unsigned)(cells - 1)); };
  // cell keys and histogram
  for (int k0 = begin + tid; k0 < n; k0 += step) {
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
      atomicAdd(count_of(m), 1);
    }
  }
  cl.sync();
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
    if (lane == 31) s_total = w;
  }
  cl.sync();
  int base = x - sum + (wid > 0 ? s_warp[wid - 1] : 0);
  for (int r = 0; r < rank; r++) base += *cl.map_shared_rank(&s_total, r);
  for (int k = c0; k < c1; k++) {
    const int v = hist[k];
    hist[k] = base;
    base += v;
  }
  cl.sync();
  // scatter
  for (int k = rank * kThreads + tid; k < n; k += nblocks * kThreads) {
    const int pos = atomicAdd(count_of(__ldcg(key + off + k)), 1);
    order[off + pos] = (int)(off + k);
  }
  cl.sync();
  // windows of the list by the whole key: bitonic sort of (key, particle)
  for (int w0 = rank * kWindow; w0 < n; w0 += nblocks * kWindow) {
    const int m = min(kWindow, n - w0);
    int size = 64;
    while (size < m) size <<= 1;
    // a warp holds elements 64 wid + lane and + 32: strides below 64 stay in its registers
    const int e0 = 64 * wid + lane, e1 = e0 + 32;
    auto element = [&](int e) -> unsigned long long {
      if (e >= m) return ~0ull;
      const int p = __ldcg(order + off + w0 + e);
      return ((unsigned long long)__ldcg(key + p) << 32) | (unsigned)p;
    };
    unsigned long long v0 = element(e0), v1 = element(e1);
    auto inner = [&](int len, int j) {  // strides j, j / 2, .. 1
      if (j == 32) {
        const bool up = (e0 & len) == 0;
        const unsigned long long lo = v0 < v1 ? v0 : v1, hi = v0 < v1 ? v1 : v0;
        v0 = up ? lo : hi;
        v1 = up ? hi : lo;
        j = 16;
      }
      for (; j > 0; j >>= 1) {
        const unsigned long long o0 = __shfl_xor_sync(0xffffffffu, v0, j), o1 = __shfl_xor_sync(0xffffffffu, v1, j);
        const bool low = (lane & j) == 0;
        if ((low == ((e0 & len) == 0)) == (o0 < v0)) v0 = o0;
        if ((low == ((e1 & len) == 0)) == (o1 < v1)) v1 = o1;
      }
    };
    for (int len = 2; len <= 64; len <<= 1) inner(len, len >> 1);
    for (int len = 128; len <= size; len <<= 1) {
      win[e0] = v0;
      win[e1] = v1;
      __syncthreads();
      for (int j = len >> 1; j > 32; j >>= 1) {
        if (tid < size / 2) {
          const int lo_k = 2 * tid - (tid & (j - 1));
          const unsigned long long u = win[lo_k], v = win[lo_k + j];
          if ((u > v) == ((lo_k & len) == 0)) {
            win[lo_k] = v;
            win[lo_k + j] = u;
          }
        }
        __syncthreads();
      }
      v0 = win[e0];
      v1 = win[e1];
      inner(len, 32);
    }
    if (e0 < m) order[off + w0 + e0] = (int)(unsigned)v0;
    if (e1 < m) order[off + w0 + e1] = (int)(unsigned)v1;
    __syncthreads();
  }
}

}  // namespace

template <class Positions>
static cudaError_t launch(const Positions& where, int nbunch, long long max_bunch, unsigned* key, int* order, cudaStream_t st) {
  const int blocks = max_bunch > kWindow ? kCluster : 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nbunch * blocks));
  cfg.blockDim = dim3(kThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)blocks;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, order_kernel<Positions>, where, key, order);
}

// loads the caller-held positions' kernel, which its first launch would otherwise do (and take device memory for)
cudaError_t load_array_order() {
  cudaFuncAttributes attr;
  return cudaFuncGetAttributes(&attr, order_kernel<ArrayPositions>);
}

cudaError_t launch_array_order(const double* x, const double* v, int n, unsigned* key, int* order, cudaStream_t st) {
  return launch(ArrayPositions{x, v, n}, 1, n, key, order, st);
}

cudaError_t launch_target_order(const DeviceState& s, unsigned* key, int* order, long long max_bunch, cudaStream_t st) {
  return launch(RingPositions{s, nullptr, 0, 0}, s.nbunch, max_bunch, key, order, st);
}

}  // namespace emppp
