// Training of the learned retarded-time proposal: one batch is one launch of train_kernel (forward, loss, backward,
// per-block weight gradients) and one of adam_kernel (sum over the blocks, Adam, the BF16 operands of the next batch).
//
// What bounds it: latency. A 4096-row batch is 0.1 GFLOP, a microsecond of the GPU if it filled it; what counts is the
// chain through the two layers and back within a block, and the two launches. So:
//   - 32 rows per block (128 blocks for a batch of 4096), eight warps per block: a warp owns 16 rows and 16 of the 64
//     hidden units, and the layers' activations pass through shared memory. The sigmoid of each hidden value is
//     evaluated once for the value and its derivative;
//   - the tensor-core operands lie in global memory as B fragments (TrainImage), one 8-byte load per lane and step;
//   - the weight gradients are FP32 as outer products in registers (each thread 4 x 4 of dW2, per row
//     two 16-byte shared loads for 16 FMAs) instead of read-modify-writes of shared memory;
//   - each block writes its partial gradient once, and adam_kernel sums the blocks in a fixed order (no atomics, so a
//     training run is reproducible), updates and rewrites the operands: no zeroing, no image launch. Each 64 rows are
//     summed by themselves, 16 after 16, and the 64s one after the other: training amplifies a last bit's difference
//     of a gradient by a hundred and more (BF16 operands that round the other way), so the sums keep the grouping that
//     trained networks so far were made with, at 0.9 us a batch more than plain sums of 32 rows;
//   - each launch starts while the one before it drains (programmatic dependent launch) and waits before it reads
//     what that one writes.
// 49 batches of 4096 rows: 2.73 ms before (64 blocks of four warps, gradients in shared memory, atomics, four launches per
// batch: 55 us each), 0.80 ms now (10.6 us a batch, and 0.28 ms of the call's own allocation, copies and waits).
//
// Rounding points (also followed by the CPU reference in oracle/mlp.py): the GEMM operands X, W1, A1 =
// silu(H1), W2 (forward) and dH2, W2 (input gradient) are rounded to BF16; products accumulate in FP32;
// biases, activations, w3 and every weight gradient are FP32.
#include "emppp_internal.cuh"
#include "mlp.cuh"

using namespace emppp;
using namespace emppp::mlp;

namespace {

constexpr int kRows = 32;       // rows of a block's tile
constexpr int kThreads = 256;   // eight warps: two 16-row halves by four groups of 16 hidden units
constexpr int kLd = 72;         // row stride of the staged activations: fragment reads of a half-warp hit 32 banks
constexpr int kGrad = 4992;     // floats between two blocks' partial gradients (4929 rounded up to whole lines)
constexpr int kAdamSlices = 8;  // threads that share the sum of one parameter
constexpr int kAdamPairs = 64;  // pairs of blocks summed per turn

// B fragments of the tensor-core passes, lane-major: entry [n-tile][k-step][lane] holds rows k = 16 kk + 2t, + 1 (x)
// and + 8, + 9 (y) of column n = 8 nt + g
struct __align__(16) TrainImage {
  uint2 w1[kH / 8][32];
  uint2 w2f[kH / 8][kH / 16][32];  // forward: k = input unit, n = output unit
  uint2 w2b[kH / 8][kH / 16][32];  // input gradient: k = output unit, n = input unit
};

// where B[k][n] lies, in 16-bit units from the start of its array
__device__ __forceinline__ int fragment_at(int k, int n) {
  const int lane = (n & 7) * 4 + ((k & 7) >> 1);
  return ((((n >> 3) * (kH / 16) + (k >> 4)) * 32 + lane) * 2 + ((k >> 3) & 1)) * 2 + (k & 1);
}

__device__ __forceinline__ unsigned short bf16_bits(float x) { return (unsigned short)(pack_bf16x2(x, 0.f) & 0xffffu); }

// writes parameter k, if it is an operand of the tensor-core passes
__device__ __forceinline__ void write_operand(TrainImage* __restrict__ img, int k, float v) {
  const unsigned short h = bf16_bits(v);
  if (k < kOffB1) {
    const int f = k / kH, u = k % kH;  // one k-step
    const int lane = (u & 7) * 4 + ((f & 7) >> 1);
    reinterpret_cast<unsigned short*>(img->w1)[(((u >> 3) * 32 + lane) * 2 + (f >> 3)) * 2 + (f & 1)] = h;
  } else if (k >= kOffW2 && k < kOffB2) {
    const int i = (k - kOffW2) / kH, o = (k - kOffW2) % kH;
    reinterpret_cast<unsigned short*>(img->w2f)[fragment_at(i, o)] = h;
    reinterpret_cast<unsigned short*>(img->w2b)[fragment_at(o, i)] = h;
  }
}

__global__ void train_image_kernel(const float* __restrict__ p, TrainImage* __restrict__ img) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < kNumParams) write_operand(img, k, p[k]);
  if (k < (kInPad - kIn) * kH) {  // padding features
    const int f = kIn + k / kH, u = k % kH;
    const int lane = (u & 7) * 4 + ((f & 7) >> 1);
    reinterpret_cast<unsigned short*>(img->w1)[(((u >> 3) * 32 + lane) * 2 + (f >> 3)) * 2 + (f & 1)] = 0;
  }
}

// programmatic dependent launch: wait for the launch before this one and its writes; let the next one start
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct __align__(16) TrainSmem {  // (rows of A1 and dH2 are read as float4)
  float A1[kRows][kLd], A2[kRows][kLd], dH1[kRows][kLd], dH2[kRows][kLd];
  float X[kRows][12];
  float z[kRows][4][kH / 8 + 1];  // the output's terms per row, fragment column pair and n-tile
  float dz[kRows];
};
static_assert(alignof(TrainSmem) >= sizeof(float4) && kLd * sizeof(float) % sizeof(float4) == 0, "float4 rows");

// rows [row0, row0 + rows) of X [m][10] and T [m]; per-block gradients of sum_r (z_r - T_r)^2 / norm
// (img and p are written by the launch that may still be running: no __restrict__, so that their loads stay behind the
// wait and go through the coherent path)
__global__ void __launch_bounds__(kThreads, 2) train_kernel(const TrainImage* img, const float* p,
                                                            const float* __restrict__ X, const float* __restrict__ T,
                                                            long long row0, long long rows, float norm, float* partial,
                                                            float* loss) {
  __shared__ TrainSmem S;
  const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, t = lane & 3, w = tid >> 5;
  const int ra = 16 * (w & 1) + g, rb = ra + 8, q = w >> 1;
  const int u2 = 4 * (tid >> 4), o2 = 4 * (tid & 15);  // this thread's 4 x 4 of dW2
  const int u1 = tid & 63, part = tid >> 6;             // this thread's column of the smaller gradients, and which
  float acc[2][4][4] = {}, gs[2][4] = {}, gb3[2] = {}, loss_acc = 0.f;  // sums by 16-row half of the tile
  if (tid < kRows) S.X[tid][10] = S.X[tid][11] = 0.f;
  bool waited = false;
  for (long long tile = blockIdx.x; tile * kRows < rows; tile += gridDim.x) {
    const long long base = row0 + tile * kRows;
    const int nr = (int)(rows - tile * kRows < kRows ? rows - tile * kRows : kRows);
    // input tile, as the GEMM sees it; the rows of X follow one another
    for (int e = tid; e < kRows * kIn; e += kThreads) S.X[e / kIn][e % kIn] = e < nr * kIn ? bf16_round(X[base * kIn + e]) : 0.f;
    const float ta = ra < nr ? T[base + ra] : 0.f, tb = rb < nr ? T[base + rb] : 0.f;
    if (!waited) {  // what the Adam step before this launch wrote: operands and parameters
      wait_for_previous();
      let_next_start();
      waited = true;
    }
    __syncthreads();
    // layer 1
    float d1[2][4], d2[2][4];
    {
      const uint32_t a[4] = {pack_bf16x2(S.X[ra][2 * t], S.X[ra][2 * t + 1]), pack_bf16x2(S.X[rb][2 * t], S.X[rb][2 * t + 1]),
                             t == 0 ? pack_bf16x2(S.X[ra][8], S.X[ra][9]) : 0u,
                             t == 0 ? pack_bf16x2(S.X[rb][8], S.X[rb][9]) : 0u};
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const int nt = 2 * q + n, o = 8 * nt + 2 * t;
        const uint2 b = img->w1[nt][lane];
        float c[4] = {0.f, 0.f, 0.f, 0.f};
        mma_bf16(c, a, b.x, b.y);
        const float2 bias = make_float2(p[kOffB1 + o], p[kOffB1 + o + 1]);
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const float h = c[k] + ((k & 1) ? bias.y : bias.x), s = sigmoid(h);
          v[k] = h * s;
          d1[n][k] = s * (1.f + h * (1.f - s));
        }
        *reinterpret_cast<float2*>(&S.A1[ra][o]) = make_float2(v[0], v[1]);
        *reinterpret_cast<float2*>(&S.A1[rb][o]) = make_float2(v[2], v[3]);
      }
    }
    __syncthreads();
    // A fragment of k-step kk of a staged activation, this warp's 16 rows
    auto fragment = [&](const float (*M)[kLd], int kk, uint32_t a[4]) {
      const int k = 16 * kk + 2 * t;
      const float2 x0 = *reinterpret_cast<const float2*>(&M[ra][k]), x1 = *reinterpret_cast<const float2*>(&M[rb][k]);
      const float2 x2 = *reinterpret_cast<const float2*>(&M[ra][k + 8]), x3 = *reinterpret_cast<const float2*>(&M[rb][k + 8]);
      a[0] = pack_bf16x2(x0.x, x0.y);
      a[1] = pack_bf16x2(x1.x, x1.y);
      a[2] = pack_bf16x2(x2.x, x2.y);
      a[3] = pack_bf16x2(x3.x, x3.y);
    };
    // layer 2 and output
    float w3[2][2];
    {
      float c[2][4] = {};
#pragma unroll
      for (int kk = 0; kk < kH / 16; kk++) {
        uint32_t a[4];
        fragment(S.A1, kk, a);
#pragma unroll
        for (int n = 0; n < 2; n++) {
          const uint2 b = img->w2f[2 * q + n][kk][lane];
          mma_bf16(c[n], a, b.x, b.y);
        }
      }
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const int nt = 2 * q + n, o = 8 * nt + 2 * t;
        const float2 bias = make_float2(p[kOffB2 + o], p[kOffB2 + o + 1]);
        w3[n][0] = p[kOffW3 + o];
        w3[n][1] = p[kOffW3 + o + 1];
        float v[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
          const float h = c[n][k] + ((k & 1) ? bias.y : bias.x), s = sigmoid(h);
          v[k] = h * s;
          d2[n][k] = s * (1.f + h * (1.f - s));
        }
        *reinterpret_cast<float2*>(&S.A2[ra][o]) = make_float2(v[0], v[1]);
        *reinterpret_cast<float2*>(&S.A2[rb][o]) = make_float2(v[2], v[3]);
        S.z[ra][t][nt] = fmaf(v[0], w3[n][0], v[1] * w3[n][1]);
        S.z[rb][t][nt] = fmaf(v[3], w3[n][1], v[2] * w3[n][0]);
      }
    }
    __syncthreads();
    // loss and dH2 = dz w3 silu'(H2)
    {
      const float b3 = p[kOffB3];
      float za = 0.f, zb = 0.f;
#pragma unroll
      for (int nt = 0; nt < kH / 8; nt++) {
        za += S.z[ra][t][nt];
        zb += S.z[rb][t][nt];
      }
      za += __shfl_xor_sync(0xffffffffu, za, 1);
      za += __shfl_xor_sync(0xffffffffu, za, 2);
      zb += __shfl_xor_sync(0xffffffffu, zb, 1);
      zb += __shfl_xor_sync(0xffffffffu, zb, 2);
      const float ea = ra < nr ? (za + b3) - ta : 0.f, eb = rb < nr ? (zb + b3) - tb : 0.f;
      const float dza = 2.f * ea / norm, dzb = 2.f * eb / norm;
      if (q == 0 && t == 0) {
        loss_acc += ea * ea + eb * eb;
        S.dz[ra] = dza;
        S.dz[rb] = dzb;
      }
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const int o = 8 * (2 * q + n) + 2 * t;
        *reinterpret_cast<float2*>(&S.dH2[ra][o]) = make_float2(dza * w3[n][0] * d2[n][0], dza * w3[n][1] * d2[n][1]);
        *reinterpret_cast<float2*>(&S.dH2[rb][o]) = make_float2(dzb * w3[n][0] * d2[n][2], dzb * w3[n][1] * d2[n][3]);
      }
    }
    __syncthreads();
    // input gradient of layer 2 on the tensor cores, dH1 = (dH2 W2^T) silu'(H1)
    {
      float c[2][4] = {};
#pragma unroll
      for (int kk = 0; kk < kH / 16; kk++) {
        uint32_t a[4];
        fragment(S.dH2, kk, a);
#pragma unroll
        for (int n = 0; n < 2; n++) {
          const uint2 b = img->w2b[2 * q + n][kk][lane];
          mma_bf16(c[n], a, b.x, b.y);
        }
      }
#pragma unroll
      for (int n = 0; n < 2; n++) {
        const int o = 8 * (2 * q + n) + 2 * t;
        *reinterpret_cast<float2*>(&S.dH1[ra][o]) = make_float2(c[n][0] * d1[n][0], c[n][1] * d1[n][1]);
        *reinterpret_cast<float2*>(&S.dH1[rb][o]) = make_float2(c[n][2] * d1[n][2], c[n][3] * d1[n][3]);
      }
    }
    // Weight gradients, 16 rows at a time: each sum of 16 starts from zero and is then added.
    // (One copy of the code for both halves: two cost 0.5 us a batch more.) dW2[u][o] += A1[r][u] dH2[r][o]
#pragma unroll 1
    for (int h = 0; h < 2; h++) {
      float c[4][4] = {};
#pragma unroll
      for (int r = 16 * h; r < 16 * h + 16; r++) {
        const float4 x = *reinterpret_cast<const float4*>(&S.A1[r][u2]), y = *reinterpret_cast<const float4*>(&S.dH2[r][o2]);
        const float xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int a = 0; a < 4; a++)
#pragma unroll
          for (int b = 0; b < 4; b++) c[a][b] += xs[a] * ys[b];
      }
#pragma unroll
      for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) {
          if (h == 0) acc[0][a][b] += c[a][b];
          else acc[1][a][b] += c[a][b];
        }
    }
    __syncthreads();
    // dW1[f][u] += X[r][f] dH1[r][u] (part p: features p, p + 4, p + 8); db1 (part 2), db2 and dw3 (part 3); db3
#pragma unroll 1
    for (int h = 0; h < 2; h++) {
      float c[4] = {};
#pragma unroll
      for (int r = 16 * h; r < 16 * h + 16; r++) {
        const float dh1 = S.dH1[r][u1];
        c[0] = fmaf(S.X[r][part], dh1, c[0]);
        c[1] = fmaf(S.X[r][part + 4], dh1, c[1]);
        if (part < 2) {
          c[2] = fmaf(S.X[r][part + 8], dh1, c[2]);
        } else if (part == 2) {
          c[2] += dh1;
        } else {
          c[2] += S.dH2[r][u1];
          c[3] = fmaf(S.A2[r][u1], S.dz[r], c[3]);
        }
      }
#pragma unroll
      for (int a = 0; a < 4; a++) {
        if (h == 0) gs[0][a] += c[a];
        else gs[1][a] += c[a];
      }
      if (tid == 0) {
        float c = 0.f;
        for (int r = 16 * h; r < 16 * h + 16; r++) c += S.dz[r];
        if (h == 0) gb3[0] += c;
        else gb3[1] += c;
      }
    }
    __syncthreads();
  }
  if (!waited) {  // no rows for this block
    wait_for_previous();
    let_next_start();
  }
  // this block's gradient: an even block's two halves are added, an odd block's follow them in adam_kernel's sum
  const bool odd = blockIdx.x & 1;
  float* out = partial + ((size_t)(blockIdx.x >> 1) * 3 + (odd ? 1 : 0)) * kGrad;
  const int u1_last = part < 2 ? kOffW1 + (part + 8) * kH + u1 : (part == 2 ? kOffB1 : kOffB2) + u1;
  if (!odd) {
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
      for (int b = 0; b < 4; b++) acc[0][a][b] += acc[1][a][b];
#pragma unroll
    for (int a = 0; a < 4; a++) gs[0][a] += gs[1][a];
    gb3[0] += gb3[1];
  }
#pragma unroll
  for (int h = 0; h < 2; h++) {
    if (h == 1 && !odd) break;
#pragma unroll
    for (int a = 0; a < 4; a++)
      *reinterpret_cast<float4*>(out + kOffW2 + (u2 + a) * kH + o2) =
          make_float4(acc[h][a][0], acc[h][a][1], acc[h][a][2], acc[h][a][3]);
    out[kOffW1 + part * kH + u1] = gs[h][0];
    out[kOffW1 + (part + 4) * kH + u1] = gs[h][1];
    out[u1_last] = gs[h][2];
    if (part == 3) out[kOffW3 + u1] = gs[h][3];
    if (tid == 0) out[kOffB3] = gb3[h];
    out += kGrad;
  }
  if (w < 2) {  // the warps of group 0 hold the rows' errors (lanes t = 0); a sum of 16 rows each
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
    if (lane == 0) atomicAdd(loss, loss_acc);
  }
}

// The sum over the blocks of parameter k's gradient, in a fixed order: the 64 rows of each pair of blocks, then pair after
// pair. The warps of a block (kAdamSlices) load and add within the pairs in turn, warp 0 adds the pairs; every lane of
// warp 0 returns its parameter's.
__device__ __forceinline__ float gradient_sum(const float* partial, int nblocks, int k) {
  __shared__ float s_sum[kAdamPairs][32];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5, npairs = (nblocks + 1) >> 1;
  float g = 0.f;
  for (int p0 = 0; p0 < npairs; p0 += kAdamPairs) {
    if (p0 > 0) __syncthreads();
    float v[kAdamPairs / kAdamSlices][3];  // all loads in flight: rows that do not exist read the first and count zero
#pragma unroll
    for (int i = 0; i < kAdamPairs / kAdamSlices; i++) {
      const int q = p0 + sl + i * kAdamSlices;
      const bool one = k < kNumParams && q < npairs, two = one && 2 * q + 1 < nblocks;
      const float* at = partial + (one ? (size_t)q * 3 * kGrad + k : 0);
      v[i][0] = __ldcg(at);
      v[i][1] = __ldcg(at + (two ? kGrad : 0));
      v[i][2] = __ldcg(at + (two ? 2 * kGrad : 0));
      if (!one) v[i][0] = 0.f;
      if (!two) v[i][1] = v[i][2] = 0.f;
    }
#pragma unroll
    for (int i = 0; i < kAdamPairs / kAdamSlices; i++) s_sum[sl + i * kAdamSlices][lane] = (v[i][0] + v[i][1]) + v[i][2];
    __syncthreads();
    if (sl == 0) {
#pragma unroll 16
      for (int q = 0; q < kAdamPairs; q++) g += s_sum[q][lane];  // (beyond npairs: zeros)
    }
  }
  return g;
}

__global__ void __launch_bounds__(32 * kAdamSlices) adam_kernel(float* p, const float* partial, int nblocks,
                                                                float* m1, float* m2, TrainImage* img, float lr, float b1, float b2, float eps, float c1,
                                                                float c2) {
  const int k = blockIdx.x * 32 + (threadIdx.x & 31);
  wait_for_previous();
  let_next_start();
  const float gk = gradient_sum(partial, nblocks, k);
  if (threadIdx.x >= 32 || k >= kNumParams) return;
  const float a = b1 * m1[k] + (1.f - b1) * gk;
  const float b = b2 * m2[k] + (1.f - b2) * gk * gk;
  m1[k] = a;
  m2[k] = b;
  const float v = p[k] - lr * (a / c1) / (sqrtf(b / c2) + eps);
  p[k] = v;
  write_operand(img, k, v);
}

__global__ void __launch_bounds__(32 * kAdamSlices) gradient_kernel(const float* __restrict__ partial, int nblocks,
                                                                    float* __restrict__ grad) {
  const int k = blockIdx.x * 32 + (threadIdx.x & 31);
  const float g = gradient_sum(partial, nblocks, k);
  if (threadIdx.x < 32 && k < kNumParams) grad[k] = g;
}

int train_blocks(long long rows, int num_sms) {
  const long long tiles = (rows + kRows - 1) / kRows;
  return (int)(tiles < 2LL * num_sms ? (tiles > 0 ? tiles : 1) : 2LL * num_sms);
}

template <class... Args>
cudaError_t launch_after(void (*kernel)(Args...), int blocks, int threads, bool overlap, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace

namespace emppp {

// device buffer of a training run: operands, then three partial gradients per pair of blocks
size_t train_buffer_bytes(long long batch_rows, int num_sms) {
  return sizeof(TrainImage) + (size_t)((train_blocks(batch_rows, num_sms) + 1) / 2 * 3) * kGrad * sizeof(float);
}

cudaError_t launch_train_image(const float* params, void* buffer, cudaStream_t st) {
  train_image_kernel<<<(kNumParams + 255) / 256, 256, 0, st>>>(params, static_cast<TrainImage*>(buffer));
  return cudaGetLastError();
}

cudaError_t launch_train_pass(void* buffer, const float* params, const float* X, const float* T, long long row0,
                              long long rows, float norm, float* loss, int num_sms, bool overlap, cudaStream_t st) {
  TrainImage* img = static_cast<TrainImage*>(buffer);
  return launch_after(train_kernel, train_blocks(rows, num_sms), kThreads, overlap, st, (const TrainImage*)img, params, X,
                      T, row0, rows, norm, reinterpret_cast<float*>(img + 1), loss);
}

cudaError_t launch_adam(float* p, void* buffer, long long rows, int num_sms, float* m1, float* m2, float lr, float b1,
                        float b2, float eps, int step, cudaStream_t st) {
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  TrainImage* img = static_cast<TrainImage*>(buffer);
  return launch_after(adam_kernel, (kNumParams + 31) / 32, 32 * kAdamSlices, true, st, p,
                      (const float*)reinterpret_cast<float*>(img + 1), train_blocks(rows, num_sms), m1, m2, img, lr, b1,
                      b2, eps, c1, c2);
}

cudaError_t launch_gradient(const void* buffer, long long rows, int num_sms, float* grad, cudaStream_t st) {
  const TrainImage* img = static_cast<const TrainImage*>(buffer);
  gradient_kernel<<<(kNumParams + 31) / 32, 32 * kAdamSlices, 0, st>>>(reinterpret_cast<const float*>(img + 1),
                                                                       train_blocks(rows, num_sms), grad);
  return cudaGetLastError();
}

}  // namespace emppp
