// kt_mlp.cu -- training and stand-alone inference kernels of the learned root-find start.
//
// Training (SIMT, FP32 accumulation): the forward pass rounds weights and activations to
// BF16 exactly as the tensor-core inference does (bf16_forward = 1), or runs in plain FP32
// (bf16_forward = 0, used to check gradients against the FP64 reference); the backward pass
// treats the rounding as the identity.  Gradients of a mini-batch are summed over row tiles in
// registers, then with one global atomic per parameter and block.  Adam updates FP32 master weights.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>

#include "../../include/kt.h"
#include "kt_mlp.cuh"

using namespace kt;

// Scratch of kt_mlp_predict_static: one packed weight set, KT_MLP_PACKED_BYTES bytes, in a
// file-scope device array.  Every GPU that loads this library holds it until the process
// exits.  In host code `g_predict_scratch` is only a host-side stand-in for the symbol: its
// device address comes from cudaGetSymbolAddress, looked up once per device and context and
// cached below.  The cache is keyed on the context's unique id as well as the device, so a
// context re-created on the same device (after cudaDeviceReset, whose new module instance may
// hold the array elsewhere) gets a fresh lookup instead of a stale address.
static __device__ __align__(256) uint32_t g_predict_scratch[kt::PK_WORDS];

namespace {
constexpr int kMaxDevices = 64;
struct ScratchAddr {
  unsigned long long ctx_id;
  uint32_t* ptr;
};
ScratchAddr g_scratch_addr[kMaxDevices] = {};
std::mutex g_scratch_mutex;

using CtxGetCurrentFn = CUresult (*)(CUcontext*);
using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);

// the unique id of the calling thread's current context (0 if there is none yet or the driver
// entry points are unavailable)
unsigned long long current_context_id() {
  static CtxGetCurrentFn get_current = nullptr;
  static CtxGetIdFn get_id = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_current = (CtxGetCurrentFn)f;
    f = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &f, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      get_id = (CtxGetIdFn)f;
  }
  CUcontext ctx = nullptr;
  unsigned long long id = 0;
  if (!get_current || !get_id || get_current(&ctx) != CUDA_SUCCESS || !ctx || get_id(ctx, &id) != CUDA_SUCCESS)
    return 0;
  return id;
}

// device address of g_predict_scratch on the current device and context (looked up on the first
// call there; cudaGetSymbolAddress allocates nothing)
int static_scratch_address(uint32_t** out) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return KT_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return KT_ERR_ARG;
  std::lock_guard<std::mutex> lock(g_scratch_mutex);
  const unsigned long long id = current_context_id();
  ScratchAddr& a = g_scratch_addr[dev];
  if (!a.ptr || id == 0 || a.ctx_id != id) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_predict_scratch);
    if (e != cudaSuccess || !p) {
      fprintf(stderr, "kt_mlp_predict_static: cudaGetSymbolAddress failed: %s\n", cudaGetErrorString(e));
      return KT_ERR_CUDA;
    }
    a.ptr = (uint32_t*)p;
    a.ctx_id = current_context_id();  // the lookup has made the device's context current
  }
  *out = a.ptr;
  return KT_OK;
}
}  // namespace

namespace {

__device__ __forceinline__ float bf16r(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// grad and loss to zero before the blocks of mlp_grad_kernel add to them; the dependent launch may start
// at once (it waits only before its first addition)
__global__ void mlp_grad_zero_kernel(float* grad, float* loss) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < MLP_NPARAM) grad[p] = 0.f;
  if (p == 0) *loss = 0.f;
}

// Gradient of the mean squared error.  A block takes tiles of 32 rows: lane = row, and each of its four
// warps eight of the 32 columns of every layer, weights broadcast from shared memory, FP32 multiply-adds
// throughout.  The activations and deltas of a tile go through shared memory (rows of 36 floats: 16-byte
// loads of consecutive rows meet no bank conflict) for the row sums: the 1,024 entries of dW2 are
// 2 x 4 per thread over the tile's rows, dW1, the biases and dW3 are spread over the threads likewise.
// All sums stay in registers over the block's tiles; one atomic per parameter and block follows.
// (Before, every thread held one row and each of the 1,313 parameters took a five-shuffle warp sum and a
// shared-memory atomic: 230 us for 8,192 rows.)  Bound by the latency of its phases: 8,192 rows are 256
// tiles, 30 MFMA in all, under a microsecond of FP32 work.
constexpr int kGradRows = 32, kGradStride = 36, kGradThreads = 128;
constexpr long long kGradBlocks = 4 * 152;  // a grid of at most four blocks per SM

template <bool BF16>
__global__ void __launch_bounds__(kGradThreads) mlp_grad_kernel(const float* __restrict__ params,
                                                                const float* __restrict__ X,
                                                                const float* __restrict__ Y, long long n, float inv_n,
                                                                float* grad, float* loss) {
  __shared__ alignas(16) float sw[MLP_NPARAM + 3];
  __shared__ alignas(16) float s_h1[kGradRows * kGradStride], s_h2[kGradRows * kGradStride],
      s_d2[kGradRows * kGradStride], s_d1[kGradRows * kGradStride];
  __shared__ float s_x[kGradRows * 8], s_y[4][kGradRows], s_dy[kGradRows];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c0 = 8 * warp;
  for (int p = tid; p < MLP_NPARAM; p += kGradThreads) {
    // biases are applied in FP32 by the tensor-core path too
    const bool bias = (p >= OFF_B1 && p < OFF_W2) || (p >= OFF_B2 && p < OFF_W3) || p == OFF_B3;
    sw[p] = (BF16 && !bias) ? bf16r(params[p]) : params[p];
  }
  const int gj = 2 * (tid >> 3), gk = 4 * (tid & 7);   // this thread's entries of dW2: rows gj, gj + 1, columns gk..gk + 3
  const int q = tid >> 5, col = lane;                  // column sums: column col over the tile's rows 8 q .. 8 q + 7
  float g2[2][4] = {}, g1[MLP_IN] = {}, gb1 = 0.f, gb2 = 0.f, g3 = 0.f, gb3 = 0.f, lsum = 0.f;
  const long long ntiles = (n + kGradRows - 1) / kGradRows;
  for (long long t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long i = t * kGradRows + lane;
    const bool valid = i < n;
    __syncthreads();  // the weights are in place; the previous tile's arrays are free
    float x[MLP_IN];
#pragma unroll
    for (int k = 0; k < MLP_IN; ++k) {
      const float v = valid ? X[i * MLP_IN + k] : 0.f;
      x[k] = BF16 ? bf16r(v) : v;
      if (warp == 0) s_x[lane * 8 + k] = x[k];
    }
    const float yt = valid ? Y[i] : 0.f;
    // layer 1
    float h[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float s = sw[OFF_B1 + c0 + j];
#pragma unroll
      for (int k = 0; k < MLP_IN; ++k) s = fmaf(sw[OFF_W1 + (c0 + j) * MLP_IN + k], x[k], s);
      s = fmaxf(s, 0.f);
      h[j] = BF16 ? bf16r(s) : s;
    }
    float4* row = reinterpret_cast<float4*>(s_h1 + lane * kGradStride + c0);
    row[0] = make_float4(h[0], h[1], h[2], h[3]);
    row[1] = make_float4(h[4], h[5], h[6], h[7]);
    __syncthreads();
    // layer 2 and this warp's share of the output
    float a[MLP_H];
#pragma unroll
    for (int k = 0; k < MLP_H; k += 4) {
      const float4 v = *reinterpret_cast<const float4*>(s_h1 + lane * kGradStride + k);
      a[k] = v.x; a[k + 1] = v.y; a[k + 2] = v.z; a[k + 3] = v.w;
    }
    float yp = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float s = sw[OFF_B2 + c0 + j];
#pragma unroll
      for (int k = 0; k < MLP_H; k += 4) {
        const float4 w = *reinterpret_cast<const float4*>(sw + OFF_W2 + (c0 + j) * MLP_H + k);
        s = fmaf(w.w, a[k + 3], fmaf(w.z, a[k + 2], fmaf(w.y, a[k + 1], fmaf(w.x, a[k], s))));
      }
      s = fmaxf(s, 0.f);
      h[j] = BF16 ? bf16r(s) : s;
      yp = fmaf(sw[OFF_W3 + c0 + j], h[j], yp);
    }
    row = reinterpret_cast<float4*>(s_h2 + lane * kGradStride + c0);
    row[0] = make_float4(h[0], h[1], h[2], h[3]);
    row[1] = make_float4(h[4], h[5], h[6], h[7]);
    s_y[warp][lane] = yp;
    __syncthreads();
    // mean squared error and the deltas of layer 2
    const float y = ((s_y[0][lane] + s_y[1][lane]) + (s_y[2][lane] + s_y[3][lane])) + sw[OFF_B3];
    const float r = valid ? (y - yt) : 0.f;
    const float dy = 2.f * r * inv_n;
    if (warp == 0) {
      s_dy[lane] = dy;
      lsum = fmaf(r * inv_n, r, lsum);
      gb3 += dy;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) h[j] = (h[j] > 0.f) ? dy * sw[OFF_W3 + c0 + j] : 0.f;
    row = reinterpret_cast<float4*>(s_d2 + lane * kGradStride + c0);
    row[0] = make_float4(h[0], h[1], h[2], h[3]);
    row[1] = make_float4(h[4], h[5], h[6], h[7]);
    __syncthreads();
    // deltas of layer 1: columns c0 .. c0 + 7 of d2 W2, gated by h1
    float d1[8] = {};
#pragma unroll
    for (int j = 0; j < MLP_H; j += 4) {
      const float4 d = *reinterpret_cast<const float4*>(s_d2 + lane * kGradStride + j);
      const float dj[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const float4 w0 = *reinterpret_cast<const float4*>(sw + OFF_W2 + (j + m) * MLP_H + c0);
        const float4 w1 = *reinterpret_cast<const float4*>(sw + OFF_W2 + (j + m) * MLP_H + c0 + 4);
        d1[0] = fmaf(dj[m], w0.x, d1[0]); d1[1] = fmaf(dj[m], w0.y, d1[1]);
        d1[2] = fmaf(dj[m], w0.z, d1[2]); d1[3] = fmaf(dj[m], w0.w, d1[3]);
        d1[4] = fmaf(dj[m], w1.x, d1[4]); d1[5] = fmaf(dj[m], w1.y, d1[5]);
        d1[6] = fmaf(dj[m], w1.z, d1[6]); d1[7] = fmaf(dj[m], w1.w, d1[7]);
      }
    }
    const float4 ha = *reinterpret_cast<const float4*>(s_h1 + lane * kGradStride + c0);
    const float4 hb = *reinterpret_cast<const float4*>(s_h1 + lane * kGradStride + c0 + 4);
    row = reinterpret_cast<float4*>(s_d1 + lane * kGradStride + c0);
    row[0] = make_float4(ha.x > 0.f ? d1[0] : 0.f, ha.y > 0.f ? d1[1] : 0.f, ha.z > 0.f ? d1[2] : 0.f,
                         ha.w > 0.f ? d1[3] : 0.f);
    row[1] = make_float4(hb.x > 0.f ? d1[4] : 0.f, hb.y > 0.f ? d1[5] : 0.f, hb.z > 0.f ? d1[6] : 0.f,
                         hb.w > 0.f ? d1[7] : 0.f);
    // dW2 over the tile's rows
#pragma unroll 8
    for (int rr = 0; rr < kGradRows; ++rr) {
      const float2 d = *reinterpret_cast<const float2*>(s_d2 + rr * kGradStride + gj);
      const float4 v = *reinterpret_cast<const float4*>(s_h1 + rr * kGradStride + gk);
      g2[0][0] = fmaf(d.x, v.x, g2[0][0]); g2[0][1] = fmaf(d.x, v.y, g2[0][1]);
      g2[0][2] = fmaf(d.x, v.z, g2[0][2]); g2[0][3] = fmaf(d.x, v.w, g2[0][3]);
      g2[1][0] = fmaf(d.y, v.x, g2[1][0]); g2[1][1] = fmaf(d.y, v.y, g2[1][1]);
      g2[1][2] = fmaf(d.y, v.z, g2[1][2]); g2[1][3] = fmaf(d.y, v.w, g2[1][3]);
    }
    __syncthreads();
    // column sums over this warp's eight rows: dW3, db2, db1, dW1
#pragma unroll
    for (int m = 0; m < kGradRows / 4; ++m) {
      const int rr = q * (kGradRows / 4) + m;
      const float d1c = s_d1[rr * kGradStride + col];
      g3 = fmaf(s_dy[rr], s_h2[rr * kGradStride + col], g3);
      gb2 += s_d2[rr * kGradStride + col];
      gb1 += d1c;
#pragma unroll
      for (int k = 0; k < MLP_IN; ++k) g1[k] = fmaf(d1c, s_x[rr * 8 + k], g1[k]);
    }
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // grad and loss are zero
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int k = 0; k < 4; ++k) atomicAdd(grad + OFF_W2 + (gj + m) * MLP_H + gk + k, g2[m][k]);
  // the four warps' column sums, combined through shared memory: [warp][entry][col]
  __syncthreads();
  float* s_c = s_h1;  // 4 x 9 x 32 floats = the size of s_h1
  float* mine = s_c + q * 9 * 32 + col;
  mine[0] = g3;
  mine[32] = gb2;
  mine[64] = gb1;
#pragma unroll
  for (int k = 0; k < MLP_IN; ++k) mine[(3 + k) * 32] = g1[k];
  __syncthreads();
  for (int p = tid; p < 9 * 32; p += kGradThreads) {
    const float v = (s_c[p] + s_c[p + 288]) + (s_c[p + 576] + s_c[p + 864]);
    const int e = p >> 5, c = p & 31;
    const int at = (e == 0) ? OFF_W3 + c : (e == 1) ? OFF_B2 + c : (e == 2) ? OFF_B1 + c : OFF_W1 + c * MLP_IN + (e - 3);
    atomicAdd(grad + at, v);
  }
  if (warp == 0) {
    const float l = warp_sum(lsum), b3 = warp_sum(gb3);
    if (lane == 0) {
      atomicAdd(loss, l);
      atomicAdd(grad + OFF_B3, b3);
    }
  }
}
static_assert(4 * 9 * 32 <= kGradRows * kGradStride, "column sums fit in s_h1");

__global__ void mlp_adam_kernel(float* params, const float* __restrict__ grad, float* m, float* v, float lr,
                                float c1, float c2) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= MLP_NPARAM) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float gp = grad[p];
  const float mp = b1 * m[p] + (1.f - b1) * gp;
  const float vp = b2 * v[p] + (1.f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  params[p] -= lr * (mp * c1) / (sqrtf(vp * c2) + eps);
}

// ---------------------------------------------------------------- training data
// The training set keeps the samples the network corrects (feature 1, r^2 = M^2/E^2, above the
// gate) in their original order, with target z = y / r^2: a stable compaction in three passes
// (per-block counts, one-block scan of the counts, per-block scatter) over tiles of
// kTgtTile samples.
constexpr int kTgtThreads = 256, kTgtPer = 4, kTgtTile = kTgtThreads * kTgtPer;

__device__ __forceinline__ bool network_corrects(const float* __restrict__ x, long long i) {
  return x[i * MLP_IN + 1] > kMlpGateR2;
}

__global__ void __launch_bounds__(kTgtThreads) targets_count_kernel(const float* __restrict__ x, long long n,
                                                                    long long* counts) {
  __shared__ int s_w[kTgtThreads / 32];
  int c = 0;
  const long long base = (long long)blockIdx.x * kTgtTile;
#pragma unroll
  for (int k = 0; k < kTgtPer; ++k) {
    const long long i = base + k * kTgtThreads + threadIdx.x;
    c += (i < n && network_corrects(x, i)) ? 1 : 0;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < kTgtThreads / 32; ++w) t += s_w[w];
    counts[blockIdx.x] = t;
  }
}

// exclusive scan of the per-block counts in place, total into *n_out (one block)
__global__ void __launch_bounds__(1024) targets_scan_kernel(long long* counts, long long nblocks, long long* n_out) {
  __shared__ long long s_part[1024];
  const long long per = (nblocks + blockDim.x - 1) / blockDim.x;
  const long long b0 = threadIdx.x * per, b1 = min(nblocks, b0 + per);
  long long t = 0;
  for (long long b = b0; b < b1; ++b) t += counts[b];
  s_part[threadIdx.x] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long acc = 0;
    for (int k = 0; k < (int)blockDim.x; ++k) {
      const long long v = s_part[k];
      s_part[k] = acc;
      acc += v;
    }
    *n_out = acc;
  }
  __syncthreads();
  long long acc = s_part[threadIdx.x];
  for (long long b = b0; b < b1; ++b) {
    const long long v = counts[b];
    counts[b] = acc;
    acc += v;
  }
}

__global__ void __launch_bounds__(kTgtThreads) targets_scatter_kernel(const float* __restrict__ x,
                                                                      const float* __restrict__ y, long long n,
                                                                      const long long* __restrict__ offsets,
                                                                      float* x_out, float* z_out) {
  __shared__ int s_w[kTgtThreads / 32];
  long long off = offsets[blockIdx.x];
  const long long base = (long long)blockIdx.x * kTgtTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < kTgtPer; ++k) {  // samples in order: row k of the tile, then the threads
    const long long i = base + k * kTgtThreads + threadIdx.x;
    const bool keep = i < n && network_corrects(x, i);
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) s_w[warp] = __popc(bal);
    __syncthreads();
    int before = 0, total = 0;
    for (int w = 0; w < kTgtThreads / 32; ++w) {
      const int c = s_w[w];
      before += (w < warp) ? c : 0;
      total += c;
    }
    if (keep) {
      const long long o = off + before + __popc(bal & ((1u << lane) - 1u));
      const float r2 = x[i * MLP_IN + 1];
#pragma unroll
      for (int m = 0; m < MLP_IN; ++m) x_out[o * MLP_IN + m] = x[i * MLP_IN + m];
      z_out[o] = __fdiv_rn(y[i], r2);
    }
    off += total;
    __syncthreads();
  }
}

// A keyed pseudo-random permutation of [0, n): a 4-round balanced Feistel network on 2h-bit
// words (4^h >= n) with a SplitMix64-finalised round function, and cycle walking back into
// [0, n).  Each walk is bounded; a walk that has not returned after kWalkMax rounds (not expected:
// at most 3/4 of the domain lies outside [0, n)) takes i itself and is flagged.
constexpr int kWalkMax = 4096;
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}
__device__ __forceinline__ unsigned long long feistel(unsigned long long v, int h, unsigned long long key) {
  const unsigned long long mask = (1ULL << h) - 1ULL;
  unsigned long long L = v >> h, R = v & mask;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const unsigned long long F = mix64(R ^ (key + 0x9e3779b97f4a7c15ULL * (unsigned long long)(r + 1))) & mask;
    const unsigned long long t = L ^ F;
    L = R;
    R = t;
  }
  return (L << h) | R;
}

__global__ void batch_kernel(const float* __restrict__ x, const float* __restrict__ y, long long n, int h,
                             unsigned long long key, long long first, long long count, float* xb, float* yb,
                             unsigned* flag) {
  const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= count) return;
  unsigned long long v = (unsigned long long)(first + k);
  int w = 0;
  do {
    v = feistel(v, h, key);
  } while (v >= (unsigned long long)n && ++w < kWalkMax);
  if (v >= (unsigned long long)n) {
    v = (unsigned long long)(first + k);
    atomicOr(flag, 1u);
  }
#pragma unroll
  for (int m = 0; m < MLP_IN; ++m) xb[k * MLP_IN + m] = x[v * MLP_IN + m];
  yb[k] = y[v];
}

}  // namespace

namespace kt {
constexpr long long kPredictBlocks = 2 * 152;  // resident at ~100 registers and 256 threads

// word i of the packed BF16 fragments + FP32 biases (see kt_mlp.cuh) of FP32 parameters
__device__ __forceinline__ uint32_t packed_word(const float* __restrict__ params, int i) {
  if (i < PK_W2) {  // W1 rows of 4 words
    const int n = i / 4, w = i % 4, k = 2 * w;
    const float lo = (k < MLP_IN) ? params[OFF_W1 + n * MLP_IN + k] : 0.f;
    const float hi = (k + 1 < MLP_IN) ? params[OFF_W1 + n * MLP_IN + k + 1] : 0.f;
    return pack_bf16x2(lo, hi);
  }
  if (i < PK_W3) {  // W2 rows of 20 words (16 used)
    const int n = (i - PK_W2) / PK_W2_STRIDE, w = (i - PK_W2) % PK_W2_STRIDE;
    return (w < 16) ? pack_bf16x2(params[OFF_W2 + n * MLP_H + 2 * w], params[OFF_W2 + n * MLP_H + 2 * w + 1]) : 0u;
  }
  if (i < PK_B1) return pack_bf16x2(params[OFF_W3 + 2 * (i - PK_W3)], params[OFF_W3 + 2 * (i - PK_W3) + 1]);
  if (i < PK_B2) return __float_as_uint(params[OFF_B1 + (i - PK_B1)]);
  if (i < PK_B3) return __float_as_uint(params[OFF_B2 + (i - PK_B2)]);
  return __float_as_uint(params[OFF_B3]);
}

__global__ void mlp_pack_kernel(const float* __restrict__ params, uint32_t* packed) {
  for (int i = threadIdx.x; i < PK_WORDS; i += blockDim.x) packed[i] = packed_word(params, i);
}

// Tensor-core inference over an array of feature rows, one launch: every block packs the weights into
// shared memory (block 0 also into the caller's scratch), every warp keeps its fragments in registers
// and walks groups of 32 rows.  A lane reads the two features its fragment holds straight from the row
// (VEC: one 8-byte load; X 8-byte aligned), a warp's load covering whole sectors, and the lanes that hold
// an output store it: no shuffles.  Bound by memory (28 B per row) and, below ~1e5 rows, by the launch.
// GPU time of 1e6 rows 17.4 us, against 4.7 + 21.1 us for a packing launch and blocks of 256 rows reading six
// scalars per lane.  (A call through the binding takes 19 us against 25, with 12% between runs.)
template <bool VEC>
__global__ void __launch_bounds__(256) mlp_predict_kernel(const float* __restrict__ params, uint32_t* scratch,
                                                          const float* __restrict__ X, long long n, float* Y) {
  __shared__ alignas(16) uint32_t sw[PK_WORDS];
  for (int i = threadIdx.x; i < PK_WORDS; i += blockDim.x) {
    const uint32_t v = packed_word(params, i);
    sw[i] = v;
    if (blockIdx.x == 0) scratch[i] = v;
  }
  __syncthreads();
  const MlpFrags f = mlp_frags(sw);
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long groups = (n + 31) / 32, warps = (long long)gridDim.x * (blockDim.x >> 5);
  auto load = [&](long long grp, float2 (&v)[2][2]) {
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long r = 32 * grp + 16 * mt + 8 * h + g;
        v[mt][h] = make_float2(0.f, 0.f);
        if (t < 3 && r < n) {
          const float* p = X + r * MLP_IN + 2 * t;
          v[mt][h] = VEC ? __ldg(reinterpret_cast<const float2*>(p)) : make_float2(__ldg(p), __ldg(p + 1));
        }
      }
  };
  long long grp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  float2 v[2][2];
  load(grp, v);
  for (; grp < groups; grp += warps) {
    float2 next[2][2];
    load(grp + warps, next);
    uint32_t a[2][2];
    float o[2][2];
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) a[mt][h] = pack_bf16x2(v[mt][h].x, v[mt][h].y);
    mlp_infer(f, a, o);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const long long r = 32 * grp + 16 * mt + 8 * h + g;
        if (t == 0 && r < n) Y[r] = o[mt][h];
        v[mt][h] = next[mt][h];
      }
  }
}

// the grid: as many blocks as are resident at once, or one warp per 32 rows
int launch_predict(const float* params, uint32_t* scratch, const float* x, long long n, float* y, cudaStream_t s) {
  const bool vec = (reinterpret_cast<uintptr_t>(x) & 7u) == 0;
  const long long want = ((n + 31) / 32 + 7) / 8;
  const unsigned grid = (unsigned)(want < kPredictBlocks ? want : kPredictBlocks);
  if (vec) mlp_predict_kernel<true><<<grid, 256, 0, s>>>(params, scratch, x, n, y);
  else mlp_predict_kernel<false><<<grid, 256, 0, s>>>(params, scratch, x, n, y);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}
}  // namespace kt

extern "C" {

int kt_mlp_predict(const float* params, const float* x, long long n, float* y, void* scratch, size_t scratch_bytes,
                   void* stream) {
  if (!params || !x || !y || n < 0 || !scratch || scratch_bytes < (size_t)KT_MLP_PACKED_BYTES) return KT_ERR_ARG;
  if (n == 0) return KT_OK;
  return kt::launch_predict(params, (uint32_t*)scratch, x, n, y, (cudaStream_t)stream);
}

int kt_mlp_predict_static(const float* params, const float* x, long long n, float* y, void* stream) {
  if (!params || !x || !y || n < 0) {
    fprintf(stderr, "kt_mlp_predict_static: null pointer or negative row count\n");
    return KT_ERR_ARG;
  }
  if (n > KT_MLP_STATIC_MAX_ROWS) {
    fprintf(stderr, "kt_mlp_predict_static: %lld rows exceed the maximum of %lld\n", n,
            (long long)KT_MLP_STATIC_MAX_ROWS);
    return KT_ERR_ARG;
  }
  if (n == 0) return KT_OK;
  uint32_t* scratch = nullptr;
  const int rc = static_scratch_address(&scratch);
  if (rc != KT_OK) return rc;
  return kt::launch_predict(params, scratch, x, n, y, (cudaStream_t)stream);
}

int kt_mlp_grad(const float* params, const float* x, const float* y_target, long long n, int bf16_forward,
                float* grad, float* loss, void* stream) {
  if (!params || !x || !y_target || !grad || !loss || n <= 0) return KT_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  mlp_grad_zero_kernel<<<(MLP_NPARAM + 255) / 256, 256, 0, s>>>(grad, loss);
  if (cudaGetLastError() != cudaSuccess) return KT_ERR_CUDA;
  // four blocks per SM hold their sums over all their tiles; programmatic launch: the forward and backward
  // passes overlap the zeroing
  const long long tiles = (n + kGradRows - 1) / kGradRows;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(tiles < kGradBlocks ? tiles : kGradBlocks));
  cfg.blockDim = dim3(kGradThreads);
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const float inv_n = (float)(1.0 / (double)n);
  const cudaError_t e = bf16_forward
                            ? cudaLaunchKernelEx(&cfg, mlp_grad_kernel<true>, params, x, y_target, n, inv_n, grad, loss)
                            : cudaLaunchKernelEx(&cfg, mlp_grad_kernel<false>, params, x, y_target, n, inv_n, grad, loss);
  return e == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

int kt_mlp_targets_workspace(long long n, size_t* bytes) {
  if (n < 0 || !bytes) return KT_ERR_ARG;
  *bytes = (size_t)((n + kTgtTile - 1) / kTgtTile + 1) * sizeof(long long);
  return KT_OK;
}

int kt_mlp_targets(const float* x, const float* y, long long n, float* x_out, float* z_out, long long* n_out,
                   void* workspace, size_t workspace_bytes, void* stream) {
  size_t need = 0;
  if (!x || !y || !x_out || !z_out || !n_out || !workspace || kt_mlp_targets_workspace(n, &need) != KT_OK ||
      workspace_bytes < need)
    return KT_ERR_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  const long long nb = (n + kTgtTile - 1) / kTgtTile;
  long long* counts = (long long*)workspace;
  if (nb == 0) return cudaMemsetAsync(n_out, 0, sizeof(long long), s) == cudaSuccess ? KT_OK : KT_ERR_CUDA;
  if (nb > 0x7fffffffLL) return KT_ERR_ARG;
  targets_count_kernel<<<(unsigned)nb, kTgtThreads, 0, s>>>(x, n, counts);
  targets_scan_kernel<<<1, 1024, 0, s>>>(counts, nb, n_out);
  targets_scatter_kernel<<<(unsigned)nb, kTgtThreads, 0, s>>>(x, y, n, counts, x_out, z_out);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

int kt_mlp_batch(const float* x, const float* y, long long n, unsigned long long seed, int epoch, long long b,
                 long long batch, float* xb, float* yb, unsigned* flag, void* stream) {
  if (!x || !y || !xb || !yb || !flag || n <= 0 || batch <= 0 || b < 0 || epoch < 0) return KT_ERR_ARG;
  const long long first = b * batch;
  if (first >= n) return KT_ERR_ARG;
  const long long count = (first + batch <= n) ? batch : n - first;
  int h = 1;
  while (h < 31 && (1LL << (2 * h)) < n) ++h;
  const unsigned long long key = seed * 0x2545f4914f6cdd1dULL + (unsigned long long)epoch;
  batch_kernel<<<(unsigned)((count + 255) / 256), 256, 0, (cudaStream_t)stream>>>(x, y, n, h, key, first, count, xb,
                                                                                    yb, flag);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

int kt_mlp_adam(float* params, const float* grad, float* m, float* v, int step, float lr, void* stream) {
  if (!params || !grad || !m || !v || step < 1 || !(lr > 0.f)) return KT_ERR_ARG;
  const double c1 = 1.0 / (1.0 - std::pow(0.9, step)), c2 = 1.0 / (1.0 - std::pow(0.999, step));
  mlp_adam_kernel<<<(KT_MLP_NPARAM + 255) / 256, 256, 0, (cudaStream_t)stream>>>(params, grad, m, v, lr, (float)c1,
                                                                                 (float)c2);
  return cudaGetLastError() == cudaSuccess ? KT_OK : KT_ERR_CUDA;
}

}  // extern "C"
