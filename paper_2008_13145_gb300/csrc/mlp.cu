// Learned selector: a 7-64-64-8 MLP performance model trained and served by
// the library's own kernels.
//
// Training (full batch): mlp_grad_kernel computes, for a chunk of samples per
// block, the forward pass, the masked squared-error gradient and the block's
// partial parameter gradient; mlp_reduce_kernel sums the partials over blocks
// in block order (deterministic) and mlp_adam_kernel applies Adam.  The three
// launches of one step are captured once in a CUDA graph and replayed, the
// Adam step counter living in device memory.
// Serving: mlp_select_kernel gives one thread per queued GEMM; the weights sit
// in shared memory and the second hidden layer is consumed unit by unit, so
// each thread keeps only 64 + 8 activations in registers.
#include <cuda_runtime.h>

#include <cmath>
#include <vector>

#include "common.cuh"

namespace ks {
namespace mlp {

constexpr int NI = 7, NH = 64, NO = 8, NP = GEMM_MLP_PARAMS;
constexpr int OW1 = 0, OB1 = OW1 + NI * NH, OW2 = OB1 + NH, OB2 = OW2 + NH * NH, OW3 = OB2 + NH, OB3 = OW3 + NH * NO;
static_assert(OB3 + NO == NP, "parameter layout");

constexpr int kChunk = 16;       // samples a training block handles at a time
constexpr int kMaxBlocks = 256;  // training blocks; each takes as many chunks as that needs
constexpr int kThreads = 256;
constexpr int kT = NH + 2;       // row pitch of the transposed W2
constexpr int kCountParts = 32;  // partial counts of the measured outputs

int grad_chunks(int n) {  // chunks per block
  const int chunks = (n + kChunk - 1) / kChunk;
  return (chunks + kMaxBlocks - 1) / kMaxBlocks;
}
int grad_blocks(int n) {
  const int per = kChunk * grad_chunks(n);
  return (n + per - 1) / per;
}

struct GradArgs {
  int n, chunks;
  const float* P;
  const float* X;
  const float* T;
  const float* mask;
  const float* count;  // kCountParts partial counts of measured outputs; unused without a mask
  float* partials;     // nblocks x NP
  float* loss_part;    // nblocks
  int* step;           // Adam step counter, incremented by block 0 (may be null)
};

// Forward pass, masked squared-error gradient and partial parameter gradient of
// a block's chunks.  Bound by shared-memory loads (about 30 MFLOP at 2,000
// samples are nothing): a warp takes two samples and its lanes two units each,
// so weights arrive as one 8-byte load per lane and activations as broadcasts of
// four, and each thread accumulates a 4 x 4 tile of W2's gradient.  W2 is kept
// transposed too: reading a column of it per lane cost a 32-way bank conflict.
// 2,000 samples, whole call: 35 us with a one-block count, chunks of 32 on 63 SMs and
// one output a thread; 18 us so, on 125 SMs (the host issues it in about that).
__global__ void __launch_bounds__(kThreads) mlp_grad_kernel(const GradArgs a) {
  extern __shared__ float sm[];
  float* P = sm;                      // NP
  float* W2T = P + NP;                // NH x kT: W2T[j][i] = W2[i][j]
  float* h1 = W2T + NH * kT;          // kChunk x NH, each layer after its ReLU
  float* h2 = h1 + kChunk * NH;       // kChunk x NH
  float* d2 = h2 + kChunk * NH;       // kChunk x NH
  float* d1 = d2 + kChunk * NH;       // kChunk x NH
  float* dy = d1 + kChunk * NH;       // kChunk x NO
  float* x = dy + kChunk * NO;        // kChunk x NI
  __shared__ float red[kThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (a.step && blockIdx.x == 0 && tid == 0) atomicAdd(a.step, 1);
  for (int p = tid; p < NP; p += kThreads) {
    const float v = a.P[p];
    P[p] = v;
    if (p >= OW2 && p < OB2) W2T[(p - OW2) % NH * kT + (p - OW2) / NH] = v;
  }
  float gw2[4][4] = {}, rest[5] = {};  // this thread's gradient entries, summed over the chunks
  float lsum = 0.f, inv = 0.f;
  for (int c = 0; c < a.chunks; ++c) {
    const int s0 = (blockIdx.x * a.chunks + c) * kChunk;
    if (s0 >= a.n) break;
    __syncthreads();  // weights stored; the last chunk's activations read
    if (tid < kChunk * NI) x[tid] = s0 + tid / NI < a.n ? a.X[(int64_t)s0 * NI + tid] : 0.f;
    __syncthreads();
    const int s = 2 * warp, j = 2 * lane;  // two samples, two units
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      float2 z = *reinterpret_cast<const float2*>(P + OB1 + j);
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const float2 w = *reinterpret_cast<const float2*>(P + OW1 + i * NH + j);
        const float xi = x[(s + u) * NI + i];
        z.x = fmaf(xi, w.x, z.x);
        z.y = fmaf(xi, w.y, z.y);
      }
      *reinterpret_cast<float2*>(h1 + (s + u) * NH + j) = make_float2(fmaxf(z.x, 0.f), fmaxf(z.y, 0.f));
    }
    __syncwarp();  // a warp reads only its own samples up to the parameter gradients
    {
      float2 z0 = *reinterpret_cast<const float2*>(P + OB2 + j), z1 = z0;
#pragma unroll 4
      for (int i = 0; i < NH; i += 4) {
        const float4 u0 = *reinterpret_cast<const float4*>(h1 + s * NH + i);
        const float4 u1 = *reinterpret_cast<const float4*>(h1 + (s + 1) * NH + i);
        const float e0[4] = {u0.x, u0.y, u0.z, u0.w}, e1[4] = {u1.x, u1.y, u1.z, u1.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 w = *reinterpret_cast<const float2*>(P + OW2 + (i + q) * NH + j);
          z0.x = fmaf(e0[q], w.x, z0.x); z0.y = fmaf(e0[q], w.y, z0.y);
          z1.x = fmaf(e1[q], w.x, z1.x); z1.y = fmaf(e1[q], w.y, z1.y);
        }
      }
      *reinterpret_cast<float2*>(h2 + s * NH + j) = make_float2(fmaxf(z0.x, 0.f), fmaxf(z0.y, 0.f));
      *reinterpret_cast<float2*>(h2 + (s + 1) * NH + j) = make_float2(fmaxf(z1.x, 0.f), fmaxf(z1.y, 0.f));
    }
    __syncwarp();
    if (c == 0) {
      // The count comes from the kernel before, which this one may overlap up to here.
      pdl_wait();
      float t = (float)a.n * NO;
      if (a.mask) {
        t = a.count[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      }
      inv = 1.f / (t > 0.f ? t : 1.f);
    }
    {  // outputs: 16 of the warp's two samples, two lanes (halves of the sum) each
      const int ss = s + (lane >> 4), o = (lane >> 1) & 7, k0 = (lane & 1) * (NH / 2), gs = s0 + ss;
      float y = (lane & 1) ? 0.f : P[OB3 + o];
#pragma unroll 8
      for (int i = k0; i < k0 + NH / 2; ++i) y = fmaf(h2[ss * NH + i], P[OW3 + i * NO + o], y);
      y += __shfl_xor_sync(0xffffffffu, y, 1);
      if (!(lane & 1)) {
        float r = 0.f;
        if (gs < a.n) {
          const float m = a.mask ? a.mask[(int64_t)gs * NO + o] : 1.f;
          r = (y - a.T[(int64_t)gs * NO + o]) * m;
        }
        lsum = fmaf(r, r, lsum);
        dy[ss * NO + o] = 2.f * r * inv;
      }
    }
    __syncwarp();
    {
      float w[2][NO];
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int o = 0; o < NO; o += 4) {
          const float4 t = *reinterpret_cast<const float4*>(P + OW3 + (j + v) * NO + o);
          w[v][o] = t.x; w[v][o + 1] = t.y; w[v][o + 2] = t.z; w[v][o + 3] = t.w;
        }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        float2 g = make_float2(0.f, 0.f);
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          const float d = dy[(s + u) * NO + o];
          g.x = fmaf(d, w[0][o], g.x);
          g.y = fmaf(d, w[1][o], g.y);
        }
        const float2 h = *reinterpret_cast<const float2*>(h2 + (s + u) * NH + j);
        *reinterpret_cast<float2*>(d2 + (s + u) * NH + j) = make_float2(h.x > 0.f ? g.x : 0.f, h.y > 0.f ? g.y : 0.f);
      }
    }
    __syncwarp();
    {
      float2 g0 = make_float2(0.f, 0.f), g1 = g0;
#pragma unroll 4
      for (int q0 = 0; q0 < NH; q0 += 4) {
        const float4 u0 = *reinterpret_cast<const float4*>(d2 + s * NH + q0);
        const float4 u1 = *reinterpret_cast<const float4*>(d2 + (s + 1) * NH + q0);
        const float e0[4] = {u0.x, u0.y, u0.z, u0.w}, e1[4] = {u1.x, u1.y, u1.z, u1.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2 w = *reinterpret_cast<const float2*>(W2T + (q0 + q) * kT + j);
          g0.x = fmaf(e0[q], w.x, g0.x); g0.y = fmaf(e0[q], w.y, g0.y);
          g1.x = fmaf(e1[q], w.x, g1.x); g1.y = fmaf(e1[q], w.y, g1.y);
        }
      }
      const float2 a0 = *reinterpret_cast<const float2*>(h1 + s * NH + j);
      const float2 a1 = *reinterpret_cast<const float2*>(h1 + (s + 1) * NH + j);
      *reinterpret_cast<float2*>(d1 + s * NH + j) = make_float2(a0.x > 0.f ? g0.x : 0.f, a0.y > 0.f ? g0.y : 0.f);
      *reinterpret_cast<float2*>(d1 + (s + 1) * NH + j) = make_float2(a1.x > 0.f ? g1.x : 0.f, a1.y > 0.f ? g1.y : 0.f);
    }
    __syncthreads();
    {
      const int i4 = 4 * (tid >> 4), j4 = 4 * (tid & 15);
#pragma unroll 4
      for (int t = 0; t < kChunk; ++t) {
        const float4 u = *reinterpret_cast<const float4*>(h1 + t * NH + i4);
        const float4 v = *reinterpret_cast<const float4*>(d2 + t * NH + j4);
        const float uu[4] = {u.x, u.y, u.z, u.w}, vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int w = 0; w < 4; ++w) gw2[q][w] = fmaf(uu[q], vv[w], gw2[q][w]);
      }
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) {  // W1, b1, b2, W3, b3 in turn
      int p = tid + k * kThreads;
      if (p >= OW2) p += NH * NH;
      if (p >= NP) continue;
      float g = rest[k];
      if (p < OB1) {
        for (int t = 0; t < kChunk; ++t) g = fmaf(x[t * NI + p / NH], d1[t * NH + p % NH], g);
      } else if (p < OW2) {
        for (int t = 0; t < kChunk; ++t) g += d1[t * NH + p - OB1];
      } else if (p < OW3) {
        for (int t = 0; t < kChunk; ++t) g += d2[t * NH + p - OB2];
      } else if (p < OB3) {
        for (int t = 0; t < kChunk; ++t) g = fmaf(h2[t * NH + (p - OW3) / NO], dy[t * NO + (p - OW3) % NO], g);
      } else {
        for (int t = 0; t < kChunk; ++t) g += dy[t * NO + p - OB3];
      }
      rest[k] = g;
    }
  }
  float* out = a.partials + (int64_t)blockIdx.x * NP;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    *reinterpret_cast<float4*>(out + OW2 + (4 * (tid >> 4) + q) * NH + 4 * (tid & 15)) =
        make_float4(gw2[q][0], gw2[q][1], gw2[q][2], gw2[q][3]);
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    int p = tid + k * kThreads;
    if (p >= OW2) p += NH * NH;
    if (p < NP) out[p] = rest[k];
  }
  // block loss partial (sum of squared masked residuals / count)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0) red[warp] = lsum;
  __syncthreads();
  if (tid == 0) {
    float t = 0.f;
    for (int w = 0; w < kThreads / 32; ++w) t += red[w];
    a.loss_part[blockIdx.x] = t * inv;
  }
}

// Sums the blocks' partials in a fixed order: 32 parameters a block, each by
// eight threads that take every eighth block's.  (One thread per parameter
// walked 63 partials in 8 us.)  Block 0 also sums the loss.
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float* partials, const float* loss_part, int nblocks,
                                                         float* grad, float* loss, float* loss_hist, const int* step,
                                                         int t0) {
  __shared__ float part[8][33];
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31, p = blockIdx.x * 32 + lane;
  pdl_wait();
  float g = 0.f;
  if (p < NP) {
#pragma unroll 8
    for (int b = q; b < nblocks; b += 8) g += partials[(int64_t)b * NP + p];
  }
  part[q][lane] = g;
  __syncthreads();
  if (q == 0) {
    if (p < NP) {
      float t = part[0][lane];
#pragma unroll
      for (int u = 1; u < 8; ++u) t += part[u][lane];
      grad[p] = t;
    }
  } else if (q == 1 && blockIdx.x == 0) {
    float l = 0.f;
    for (int b = lane; b < nblocks; b += 32) l += loss_part[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) {
      if (loss) *loss = l;
      if (loss_hist && step) loss_hist[*step - t0 - 1] = l;
    }
  }
}

// Partial sums of the mask, one per block of the kCountParts that the gradient kernel adds.
__global__ void __launch_bounds__(256) mlp_count_kernel(const float* mask, int64_t total, float* count) {
  __shared__ float red[8];
  pdl_launch_dependents();  // the gradient kernel's forward pass reads nothing that is written here
  float c = 0.f;
  const int64_t each = (total + kCountParts - 1) / kCountParts, first = blockIdx.x * each;
  const int64_t last = first + each < total ? first + each : total;
#pragma unroll 4
  for (int64_t i = first + threadIdx.x; i < last; i += blockDim.x) c += mask[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < 8; ++w) t += red[w];
    count[blockIdx.x] = t;
  }
}

__global__ void mlp_adam_kernel(float* P, const float* g, float* m, float* v, const int* step_dev, int step_host,
                                float lr, float b1, float b2, float eps) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= NP) return;
  const int t = step_dev ? *step_dev : step_host;
  const float gp = g[p];
  const float mp = b1 * m[p] + (1.f - b1) * gp;
  const float vp = b2 * v[p] + (1.f - b2) * gp * gp;
  m[p] = mp;
  v[p] = vp;
  const float mh = mp / (1.f - powf(b1, (float)t));
  const float vh = vp / (1.f - powf(b2, (float)t));
  P[p] -= lr * mh / (sqrtf(vh) + eps);
}

__device__ __forceinline__ float feature(int q, const int64_t* sh) {
  switch (q) {
    case 0: return log2f((float)sh[0]) / 12.f;
    case 1: return log2f((float)sh[1]) / 12.f;
    case 2: return log2f((float)sh[2]) / 12.f;
    case 3: return log2f((float)sh[3]) / 4.f;
    case 4: return (float)sh[4];
    case 5: return (float)sh[5];
    default: return (float)sh[6] / 3.f;
  }
}

// Training targets: per row of an n x d throughput table, log(perf / row max)
// over the measured (perf > 0) entries, 0 elsewhere, and the mask of measured
// entries (a row with none measured is all masked).
__global__ void mlp_targets_kernel(int n, int d, const float* perf, float* T, float* mask) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  const float* p = perf + (int64_t)r * d;
  float mx = 0.f;
  for (int j = 0; j < d; ++j) mx = fmaxf(mx, p[j]);
  for (int j = 0; j < d; ++j) {
    const bool ok = p[j] > 0.f;
    T[(int64_t)r * d + j] = ok ? logf(p[j] / mx) : 0.f;
    mask[(int64_t)r * d + j] = ok ? 1.f : 0.f;
  }
}

__global__ void mlp_features_kernel(int n, const int64_t* shapes, float* X) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
#pragma unroll
  for (int q = 0; q < NI; ++q) X[(int64_t)r * NI + q] = feature(q, shapes + (int64_t)r * 7);
}

// One thread per row: y = network(x); optionally pick argmax over the first n_out outputs.
template <bool FROM_SHAPES>
__global__ void __launch_bounds__(128) mlp_forward_kernel(int n, const float* Pg, const float* X, const int64_t* shapes,
                                                          float* Y, int n_out, const int32_t* ids, int32_t* ids_out) {
  __shared__ float P[NP];
  for (int p = threadIdx.x; p < NP; p += blockDim.x) P[p] = Pg[p];
  __syncthreads();
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  float x[NI];
#pragma unroll
  for (int i = 0; i < NI; ++i) x[i] = FROM_SHAPES ? feature(i, shapes + (int64_t)r * 7) : X[(int64_t)r * NI + i];
  float h1[NH];
#pragma unroll
  for (int j = 0; j < NH; ++j) {
    float z = P[OB1 + j];
#pragma unroll
    for (int i = 0; i < NI; ++i) z = fmaf(x[i], P[OW1 + i * NH + j], z);
    h1[j] = fmaxf(z, 0.f);
  }
  float y[NO];
#pragma unroll
  for (int o = 0; o < NO; ++o) y[o] = P[OB3 + o];
#pragma unroll 1
  for (int j = 0; j < NH; ++j) {
    float z = P[OB2 + j];
#pragma unroll
    for (int i = 0; i < NH; ++i) z = fmaf(h1[i], P[OW2 + i * NH + j], z);
    const float h = fmaxf(z, 0.f);
#pragma unroll
    for (int o = 0; o < NO; ++o) y[o] = fmaf(h, P[OW3 + j * NO + o], y[o]);
  }
  if (Y) {
#pragma unroll
    for (int o = 0; o < NO; ++o) Y[(int64_t)r * NO + o] = y[o];
  }
  if (ids_out) {
    int best = 0;
    for (int o = 1; o < n_out; ++o)
      if (y[o] > y[best]) best = o;
    ids_out[r] = ids[best];
  }
}

struct Ids {
  int32_t v[GEMM_MAX_DEPLOYED];
};

gemm_status_t fail(cudaError_t e) {
  set_last_cuda_error(e);
  return GEMM_ERR_CUDA;
}

constexpr size_t kGradSmem = sizeof(float) * (NP + NH * kT + kChunk * (4 * NH + NO + NI));

cudaError_t ensure_attr() {
  static unsigned long long done = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  const unsigned long long bit = 1ull << (dev & 63);
  if (__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGradSmem);
  if (e == cudaSuccess) __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
  return e;
}

// Scratch for one training configuration: partials, loss partials, count, grad, loss, step.
struct Workspace {
  float* partials;
  float* loss_part;
  float* count;
  float* grad;
  float* loss;
  int* step;
  char* base;
};

cudaError_t ws_alloc(int nblocks, cudaStream_t s, Workspace* w) {
  const size_t bytes = sizeof(float) * ((size_t)nblocks * NP + nblocks + kCountParts + NP + 1) + sizeof(int) + 6 * 256;
  cudaError_t e = scratch_alloc(reinterpret_cast<void**>(&w->base), bytes, s);
  if (e != cudaSuccess) return e;
  char* p = w->base;
  auto carve = [&](size_t nb) {
    char* r = p;
    p += (nb + 255) / 256 * 256;
    return r;
  };
  w->partials = reinterpret_cast<float*>(carve(sizeof(float) * (size_t)nblocks * NP));
  w->loss_part = reinterpret_cast<float*>(carve(sizeof(float) * nblocks));
  w->count = reinterpret_cast<float*>(carve(sizeof(float) * kCountParts));
  w->grad = reinterpret_cast<float*>(carve(sizeof(float) * NP));
  w->loss = reinterpret_cast<float*>(carve(sizeof(float)));
  w->step = reinterpret_cast<int*>(carve(sizeof(int)));
  return cudaSuccess;
}

// ---------------------------------------------------------------- allocation-free loss/gradient
// Scratch of mlp_loss_grad_noalloc: per-block gradient partials for up to
// kNoAllocMaxSamples samples, then the per-block losses, then the counts of
// measured outputs.  Every device that loads the library holds this array
// (about 5.3 MB) until the process exits.
constexpr int kNoAllocMaxSamples = 8192;
constexpr int kNoAllocMaxBlocks = kMaxBlocks;
static_assert(kCountParts <= 64, "the scratch holds 64 floats after the losses");
constexpr size_t kNoAllocFloats = (size_t)kNoAllocMaxBlocks * NP + kNoAllocMaxBlocks + 64;
static __device__ __align__(256) float g_noalloc_scratch[kNoAllocFloats];

// Device address of the scratch array on the current device.  In host code
// g_noalloc_scratch names a host-side stand-in, so the address is looked up
// once per device and cached.
float* noalloc_scratch(cudaError_t* err) {
  static float* addr[64] = {nullptr};
  static std::mutex mu;
  int dev = 0;
  *err = cudaGetDevice(&dev);
  if (*err != cudaSuccess) return nullptr;
  if (dev < 0 || dev >= 64) {
    *err = cudaErrorInvalidDevice;
    return nullptr;
  }
  std::lock_guard<std::mutex> g(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    *err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (*err != cudaSuccess) return nullptr;
    addr[dev] = static_cast<float*>(p);
  }
  return addr[dev];
}

// The gradient kernels of one pass: the count of measured outputs (without a mask
// it is known), the blocks' partials, their sums.  Each may start while the one
// before it drains; all writes and all reads of what those write come after
// the wait.
cudaError_t launch_count(const float* mask, int n, float* count, cudaStream_t s) {
  if (!mask) return cudaSuccess;
  mlp_count_kernel<<<kCountParts, 256, 0, s>>>(mask, (int64_t)n * NO, count);
  return cudaGetLastError();
}
cudaError_t launch_grad(const GradArgs& a, float* grad, float* loss, float* loss_hist, int t0, bool overlap,
                        cudaStream_t s) {
  const int nb = grad_blocks(a.n);
  cudaError_t e = cudaSuccess;
  if (overlap) {
    e = launch_pdl(mlp_grad_kernel, dim3(nb), dim3(kThreads), kGradSmem, s, nullptr, 0, a);
  } else {
    mlp_grad_kernel<<<nb, kThreads, kGradSmem, s>>>(a);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  return launch_pdl(mlp_reduce_kernel, dim3((NP + 31) / 32), dim3(256), 0, s, nullptr, 0,
                    static_cast<const float*>(a.partials), static_cast<const float*>(a.loss_part), nb, grad, loss,
                    loss_hist, static_cast<const int*>(a.step), t0);
}

}  // namespace mlp
}  // namespace ks

using namespace ks;
using namespace ks::mlp;

extern "C" {

gemm_status_t mlp_features(int32_t n, const int64_t* shapes, float* X, void* stream) {
  if (n < 0 || (n > 0 && (!shapes || !X))) return GEMM_ERR_INVALID_ARG;
  if (n == 0) return GEMM_OK;
  mlp_features_kernel<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, shapes, X);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_targets(int32_t n, int32_t d, const float* perf, float* T, float* mask, void* stream) {
  if (n < 0 || d < 1 || (n > 0 && (!perf || !T || !mask))) return GEMM_ERR_INVALID_ARG;
  if (n == 0) return GEMM_OK;
  mlp_targets_kernel<<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, d, perf, T, mask);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_forward(int32_t n, const float* P, const float* X, float* Y, void* stream) {
  if (n < 0 || (n > 0 && (!P || !X || !Y))) return GEMM_ERR_INVALID_ARG;
  if (n == 0) return GEMM_OK;
  mlp_forward_kernel<false><<<(n + 127) / 128, 128, 0, static_cast<cudaStream_t>(stream)>>>(n, P, X, nullptr, Y, 0,
                                                                                            nullptr, nullptr);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_loss_grad(int32_t n, const float* P, const float* X, const float* T, const float* mask,
                            float* grad, float* loss, void* stream) {
  if (n < 1 || !P || !X || !T || !grad || !loss) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = ensure_attr();
  if (e != cudaSuccess) return fail(e);
  Workspace w;
  if ((e = ws_alloc(grad_blocks(n), s, &w)) != cudaSuccess) return fail(e);
  GradArgs a{n, grad_chunks(n), P, X, T, mask, w.count, w.partials, w.loss_part, nullptr};
  e = launch_count(mask, n, w.count, s);
  if (e == cudaSuccess) e = launch_grad(a, grad, loss, nullptr, 0, mask != nullptr, s);
  cudaFreeAsync(w.base, s);
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_loss_grad_noalloc(int32_t n, const float* P, const float* X, const float* T, const float* mask,
                                    float* grad, float* loss, void* stream) {
  if (n < 1 || !P || !X || !T || !grad || !loss) return GEMM_ERR_INVALID_ARG;
  if (n > kNoAllocMaxSamples) return GEMM_ERR_UNSUPPORTED;  // beyond the static scratch
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = ensure_attr();
  if (e != cudaSuccess) return fail(e);
  float* base = noalloc_scratch(&e);
  if (!base) return fail(e);
  float* partials = base;
  float* loss_part = base + (size_t)kNoAllocMaxBlocks * NP;
  float* count = loss_part + kNoAllocMaxBlocks;
  // Every scratch value read below is written earlier in this call (the counts,
  // then the partials and losses of the blocks), so nothing needs clearing.
  GradArgs a{n, grad_chunks(n), P, X, T, mask, count, partials, loss_part, nullptr};
  e = launch_count(mask, n, count, s);
  if (e == cudaSuccess) e = launch_grad(a, grad, loss, nullptr, 0, mask != nullptr, s);
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_adam_step(float* P, const float* g, float* m, float* v, int32_t t, float lr, float b1, float b2,
                            float eps, void* stream) {
  if (!P || !g || !m || !v || t < 1 || !(lr > 0.f)) return GEMM_ERR_INVALID_ARG;
  mlp_adam_kernel<<<(NP + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(P, g, m, v, nullptr, t, lr, b1,
                                                                                   b2, eps);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t mlp_train(int32_t n, float* P, const float* X, const float* T, const float* mask, float* m, float* v,
                        int32_t t0, int32_t steps, float lr, float b1, float b2, float eps, float* loss_hist,
                        void* stream) {
  if (n < 1 || !P || !X || !T || !m || !v || t0 < 0 || steps < 0 || !(lr > 0.f)) return GEMM_ERR_INVALID_ARG;
  if (steps == 0) return GEMM_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = ensure_attr();
  if (e != cudaSuccess) return fail(e);
  Workspace w;
  if ((e = ws_alloc(grad_blocks(n), s, &w)) != cudaSuccess) return fail(e);
  e = launch_count(mask, n, w.count, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(w.step, &t0, sizeof(int), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaStream_t cap = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    GradArgs a{n, grad_chunks(n), P, X, T, mask, w.count, w.partials, w.loss_part, w.step};
    cudaError_t el = launch_grad(a, w.grad, w.loss, loss_hist, t0, false, cap);
    mlp_adam_kernel<<<(NP + 255) / 256, 256, 0, cap>>>(P, w.grad, m, v, w.step, 0, lr, b1, b2, eps);
    cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
    e = (e2 != cudaSuccess) ? e2 : el != cudaSuccess ? el : cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaGraphInstantiate(&exec, graph, 0);
  for (int i = 0; i < steps && e == cudaSuccess; ++i) e = cudaGraphLaunch(exec, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (exec) cudaGraphExecDestroy(exec);
  if (graph) cudaGraphDestroy(graph);
  if (cap) cudaStreamDestroy(cap);
  cudaFreeAsync(w.base, s);
  cudaStreamSynchronize(s);
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

gemm_status_t select_kernels_batched(gemm_handle_t h, int32_t n, const int64_t* shapes, int32_t* ids_out,
                                     float* pred, void* stream) {
  if (!h || n < 0 || (n > 0 && (!shapes || !ids_out))) return GEMM_ERR_INVALID_ARG;
  if (h->mlp.empty()) return GEMM_ERR_UNSUPPORTED;
  if ((int)h->ids.size() > NO) return GEMM_ERR_UNSUPPORTED;
  if (n == 0) return GEMM_OK;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 64) return fail(e);
  float* P = nullptr;
  {
    std::lock_guard<std::mutex> g(h->dev_mu);
    if (!h->dev_mlp[dev]) {
      float* p = nullptr;
      if ((e = cudaMalloc(&p, sizeof(float) * NP)) != cudaSuccess) return fail(e);
      if ((e = cudaMemcpy(p, h->mlp.data(), sizeof(float) * NP, cudaMemcpyHostToDevice)) != cudaSuccess) {
        cudaFree(p);
        return fail(e);
      }
      h->dev_mlp[dev] = p;
    }
    P = h->dev_mlp[dev];
  }
  Ids ids{};
  for (size_t i = 0; i < h->ids.size(); ++i) ids.v[i] = h->ids[i];
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int32_t* dids = nullptr;
  if ((e = cudaMallocAsync(reinterpret_cast<void**>(&dids), sizeof(ids.v), s)) != cudaSuccess) return fail(e);
  e = cudaMemcpyAsync(dids, ids.v, sizeof(ids.v), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) {
    mlp_forward_kernel<true><<<(n + 127) / 128, 128, 0, s>>>(n, P, nullptr, shapes, pred, (int)h->ids.size(), dids,
                                                           ids_out);
    e = cudaGetLastError();
  }
  cudaFreeAsync(dids, s);
  return e == cudaSuccess ? GEMM_OK : fail(e);
}

}  // extern "C"
