// The layers around the GEMMs of a convolutional network (Section 6: VGG16
// inference with the library's matrix multiply).  Activations are NHWC, so a
// 3x3 convolution is im2col (rows = output pixels, columns = (kh, kw, c))
// times the weights (Cout x 9 Cin, i.e. op(B) = B^T), and the GEMM's output
// rows are already the next NHWC activation.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>

#include "common.cuh"

namespace ks {
namespace {

// out[(n, h, w), (kh * 3 + kw) * C + c] = x[n, h + kh - 1, w + kw - 1, c], zero outside.
// V = 4 moves 4 channels per thread (C % 4 == 0, 16-byte aligned rows); the
// index type I is 32-bit whenever the element count allows, which keeps the
// per-element index arithmetic cheap on this memory-bound copy.
template <int V, typename I>
__global__ void im2col3x3_kernel(const float* __restrict__ x, int N, int H, int W, int C, float* __restrict__ out,
                                 int64_t ld) {
  const int CV = C / V;
  const I per_row = (I)9 * CV;
  const I total = (I)N * H * W * per_row;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
    const I row = t / per_row;
    const int q = (int)(t - row * per_row);
    const int tap = q / CV, c = (q - tap * CV) * V;
    const int kh = tap / 3, kw = tap - kh * 3;
    const I hw = row % ((I)H * W);
    const int n = (int)(row / ((I)H * W)), h = (int)(hw / W), w = (int)(hw - (I)h * W);
    const int hh = h + kh - 1, ww = w + kw - 1;
    float* dst = out + (int64_t)row * ld + tap * C + c;
    const bool inside = hh >= 0 && hh < H && ww >= 0 && ww < W;
    const float* src = x + (((int64_t)n * H + hh) * W + ww) * C + c;
    if constexpr (V == 4) {
      *reinterpret_cast<float4*>(dst) = inside ? __ldg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
    } else {
      *dst = inside ? __ldg(src) : 0.f;
    }
  }
}

// y[r, j] = act(y[r, j] + bias[j]) over rows x cols with leading dimension ld, V columns per thread.
template <int V, typename I>
__global__ void bias_act_kernel(float* y, int64_t rows, int cols, int64_t ld, const float* bias, int relu) {
  const int cv = cols / V;
  const I total = (I)rows * cv;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
    const I r = t / cv;
    const int j = (int)(t - r * cv) * V;
    float* p = y + (int64_t)r * ld + j;
    if constexpr (V == 4) {
      float4 v = *reinterpret_cast<float4*>(p);
      if (bias) {
        const float4 b = __ldg(reinterpret_cast<const float4*>(bias + j));
        v.x += b.x; v.y += b.y; v.z += b.z; v.w += b.w;
      }
      if (relu) { v.x = fmaxf(v.x, 0.f); v.y = fmaxf(v.y, 0.f); v.z = fmaxf(v.z, 0.f); v.w = fmaxf(v.w, 0.f); }
      *reinterpret_cast<float4*>(p) = v;
    } else {
      float v = *p + (bias ? bias[j] : 0.f);
      if (relu) v = fmaxf(v, 0.f);
      *p = v;
    }
  }
}

// 2 x 2, stride 2 max pooling of NHWC x (H, W even), V channels per thread.
template <int V, typename I>
__global__ void maxpool2x2_kernel(const float* __restrict__ x, int N, int H, int W, int C, float* __restrict__ out) {
  const int Ho = H / 2, Wo = W / 2, CV = C / V;
  const I total = (I)N * Ho * Wo * CV;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
    const I p = t / CV;
    const int c = (int)(t - p * CV) * V;
    const I hw = p % ((I)Ho * Wo);
    const int n = (int)(p / ((I)Ho * Wo)), ho = (int)(hw / Wo), wo = (int)(hw - (I)ho * Wo);
    const float* b = x + (((int64_t)n * H + 2 * ho) * W + 2 * wo) * C + c;
    const int64_t rs = (int64_t)W * C;
    if constexpr (V == 4) {
      const float4 a0 = __ldg(reinterpret_cast<const float4*>(b)), a1 = __ldg(reinterpret_cast<const float4*>(b + C));
      const float4 a2 = __ldg(reinterpret_cast<const float4*>(b + rs));
      const float4 a3 = __ldg(reinterpret_cast<const float4*>(b + rs + C));
      *reinterpret_cast<float4*>(out + (int64_t)p * C + c) =
          make_float4(fmaxf(fmaxf(a0.x, a1.x), fmaxf(a2.x, a3.x)), fmaxf(fmaxf(a0.y, a1.y), fmaxf(a2.y, a3.y)),
                      fmaxf(fmaxf(a0.z, a1.z), fmaxf(a2.z, a3.z)), fmaxf(fmaxf(a0.w, a1.w), fmaxf(a2.w, a3.w)));
    } else {
      out[(int64_t)p * C + c] = fmaxf(fmaxf(b[0], b[C]), fmaxf(b[rs], b[rs + C]));
    }
  }
}

// The same im2col from NCHW activations (the GEMM-batched layout of Section 6,
// where each image's output is Cout x (H W)): out[(n, h, w), (kh * 3 + kw) * C + c]
// = x[n, c, h + kh - 1, w + kw - 1].  Consecutive threads write consecutive columns.
template <typename I>
__global__ void im2col3x3_nchw_kernel(const float* __restrict__ x, int N, int C, int H, int W,
                                      float* __restrict__ out, int64_t ld) {
  const I per_row = (I)9 * C;
  const I total = (I)N * H * W * per_row;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
    const I row = t / per_row;
    const int q = (int)(t - row * per_row);
    const int tap = q / C, c = q - tap * C;
    const int kh = tap / 3, kw = tap - kh * 3;
    const I hw = row % ((I)H * W);
    const int n = (int)(row / ((I)H * W)), h = (int)(hw / W), w = (int)(hw - (I)h * W);
    const int hh = h + kh - 1, ww = w + kw - 1;
    const bool inside = hh >= 0 && hh < H && ww >= 0 && ww < W;
    out[(int64_t)row * ld + q] = inside ? __ldg(x + (((int64_t)n * C + c) * H + hh) * W + ww) : 0.f;
  }
}

// y[n, c, p] = act(y[n, c, p] + bias[c]) for NCHW activations (p over H W).
template <typename I>
__global__ void bias_act_nchw_kernel(float* y, int N, int C, int64_t HW, const float* bias, int relu) {
  const I total = (I)N * C * HW;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (I)gridDim.x * blockDim.x) {
    const int c = (int)((t / (I)HW) % C);
    float v = y[t] + (bias ? __ldg(bias + c) : 0.f);
    if (relu) v = fmaxf(v, 0.f);
    y[t] = v;
  }
}

// 3 x 3 convolution (padding 1) of an NHWC image of C <= 4 channels with bias and
// ReLU: the first layer of a network, whose product has K = 9 C.  Bound by writing
// the result and by its FMAs (205 MB and 1.4 G for VGG16's first layer on 16
// images).  A thread has four neighbouring positions and eight outputs, so an image
// value serves eight FMAs and a weight, broadcast from shared memory, four; the
// eight lanes of a position write 256 consecutive bytes.  The sum over K runs in
// the column order of im2col.  VGG16's first layer, 16 images: 113 us against 255
// as im2col, product and bias + ReLU (16 outputs a thread: 138, one block an SM).
constexpr int kFewPx = 4, kFewOut = 8, kFewThreads = 256;
template <int C>
__global__ void __launch_bounds__(kFewThreads) conv3x3_few_kernel(const float* __restrict__ x, int64_t quads, int H,
                                                                  int W, const float* __restrict__ w, int Cout,
                                                                  const float* __restrict__ bias, int relu,
                                                                  float* __restrict__ out) {
  extern __shared__ float4 ws4[];  // 9 C x Cout
  float* ws = reinterpret_cast<float*>(ws4);
  for (int i = threadIdx.x; i < 9 * C * Cout; i += kFewThreads) ws[i % (9 * C) * Cout + i / (9 * C)] = w[i];
  __syncthreads();
  const int groups = Cout / kFewOut;
  for (int64_t t = (int64_t)blockIdx.x * kFewThreads + threadIdx.x; t < quads * groups;
       t += (int64_t)gridDim.x * kFewThreads) {
    const int64_t quad = t / groups, m = quad * kFewPx;
    const int o0 = (int)(t - quad * groups) * kFewOut;
    const int hw = (int)(m % ((int64_t)H * W)), h = hw / W, w0 = hw - h * W;
    float acc[kFewPx][kFewOut];
#pragma unroll
    for (int p = 0; p < kFewPx; ++p)
#pragma unroll
      for (int o = 0; o < kFewOut; ++o) acc[p][o] = 0.f;
#pragma unroll
    for (int kh = 0; kh < 3; ++kh) {
      float v[(kFewPx + 2) * C];  // the row's six positions
      const bool row = h + kh >= 1 && h + kh <= H;
      const float* src = x + (m + (int64_t)(kh - 1) * W - 1) * C;
#pragma unroll
      for (int i = 0; i < (kFewPx + 2) * C; ++i) {
        const int col = w0 - 1 + i / C;
        v[i] = row && col >= 0 && col < W ? __ldg(src + i) : 0.f;
      }
#pragma unroll
      for (int kw = 0; kw < 3; ++kw)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const float4* wk = reinterpret_cast<const float4*>(ws + ((kh * 3 + kw) * C + c) * Cout + o0);
#pragma unroll
          for (int q = 0; q < kFewOut / 4; ++q) {
            const float4 u = wk[q];
#pragma unroll
            for (int p = 0; p < kFewPx; ++p) {
              const float a = v[(p + kw) * C + c];
              acc[p][4 * q] = fmaf(a, u.x, acc[p][4 * q]);
              acc[p][4 * q + 1] = fmaf(a, u.y, acc[p][4 * q + 1]);
              acc[p][4 * q + 2] = fmaf(a, u.z, acc[p][4 * q + 2]);
              acc[p][4 * q + 3] = fmaf(a, u.w, acc[p][4 * q + 3]);
            }
          }
        }
    }
#pragma unroll
    for (int q = 0; q < kFewOut / 4; ++q) {
      const float4 b = bias ? __ldg(reinterpret_cast<const float4*>(bias + o0) + q) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int p = 0; p < kFewPx; ++p) {
        float4 y = make_float4(acc[p][4 * q] + b.x, acc[p][4 * q + 1] + b.y, acc[p][4 * q + 2] + b.z,
                               acc[p][4 * q + 3] + b.w);
        if (relu) y = make_float4(fmaxf(y.x, 0.f), fmaxf(y.y, 0.f), fmaxf(y.z, 0.f), fmaxf(y.w, 0.f));
        *reinterpret_cast<float4*>(out + (m + p) * Cout + o0 + 4 * q) = y;
      }
    }
  }
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

int grid_for(int64_t total) {
  const int64_t b = (total + 255) / 256;
  return (int)(b < 152 * 32 ? (b < 1 ? 1 : b) : 152 * 32);
}

gemm_status_t done(cudaError_t e) {
  if (e == cudaSuccess) return GEMM_OK;
  set_last_cuda_error(e);
  return GEMM_ERR_CUDA;
}
}  // namespace

// Whether conv3x3_few takes this layer: few channels, rows of whole position
// quads, outputs in whole groups, 16-byte rows, and enough positions that its
// blocks do not mostly load weights.
bool conv3x3_few_takes(int N, int H, int W, int C, int Cout, const float* bias, const float* out) {
  return C <= 4 && W % kFewPx == 0 && Cout % kFewOut == 0 && Cout <= 256 && aligned16(out) &&
         (!bias || aligned16(bias)) && (int64_t)N * H * W >= 152 * 64;
}

cudaError_t conv3x3_few(const float* x, int N, int H, int W, int C, const float* w, int Cout, const float* bias,
                        int relu, float* out, cudaStream_t s) {
  const int64_t quads = (int64_t)N * H * W / kFewPx, threads = quads * (Cout / kFewOut);
  const int grid = (int)std::min<int64_t>((threads + kFewThreads - 1) / kFewThreads, 152 * 8);
  const size_t smem = (size_t)9 * C * Cout * sizeof(float);  // at most 36,864 bytes
  switch (C) {
    case 1: conv3x3_few_kernel<1><<<grid, kFewThreads, smem, s>>>(x, quads, H, W, w, Cout, bias, relu, out); break;
    case 2: conv3x3_few_kernel<2><<<grid, kFewThreads, smem, s>>>(x, quads, H, W, w, Cout, bias, relu, out); break;
    case 3: conv3x3_few_kernel<3><<<grid, kFewThreads, smem, s>>>(x, quads, H, W, w, Cout, bias, relu, out); break;
    default: conv3x3_few_kernel<4><<<grid, kFewThreads, smem, s>>>(x, quads, H, W, w, Cout, bias, relu, out); break;
  }
  return cudaGetLastError();
}
}  // namespace ks

using namespace ks;

extern "C" {

gemm_status_t kselect_im2col3x3(const float* x, int32_t N, int32_t H, int32_t W, int32_t C, float* out, int64_t ld,
                                void* stream) {
  if (N < 0 || H < 0 || W < 0 || C < 1 || ld < 9LL * C) return GEMM_ERR_INVALID_ARG;
  const int64_t total = (int64_t)N * H * W * 9 * C;
  if (total == 0) return GEMM_OK;
  if (!x || !out) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = C % 4 == 0 && ld % 4 == 0 && aligned16(x) && aligned16(out);
  const int64_t work = vec ? total / 4 : total;
  const bool small = work < ((int64_t)1 << 31) - 152LL * 32 * 256;
  if (vec && small) im2col3x3_kernel<4, int32_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out, ld);
  else if (vec) im2col3x3_kernel<4, int64_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out, ld);
  else if (small) im2col3x3_kernel<1, int32_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out, ld);
  else im2col3x3_kernel<1, int64_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out, ld);
  return done(cudaGetLastError());
}

gemm_status_t kselect_bias_act(float* y, int64_t rows, int32_t cols, int64_t ld, const float* bias, int32_t relu,
                               void* stream) {
  if (rows < 0 || cols < 0 || ld < cols) return GEMM_ERR_INVALID_ARG;
  if (rows == 0 || cols == 0) return GEMM_OK;
  if (!y) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = cols % 4 == 0 && ld % 4 == 0 && aligned16(y) && (!bias || aligned16(bias));
  const int64_t work = vec ? rows * (cols / 4) : rows * cols;
  const bool small = work < ((int64_t)1 << 31) - 152LL * 32 * 256;
  if (vec && small) bias_act_kernel<4, int32_t><<<grid_for(work), 256, 0, s>>>(y, rows, cols, ld, bias, relu);
  else if (vec) bias_act_kernel<4, int64_t><<<grid_for(work), 256, 0, s>>>(y, rows, cols, ld, bias, relu);
  else if (small) bias_act_kernel<1, int32_t><<<grid_for(work), 256, 0, s>>>(y, rows, cols, ld, bias, relu);
  else bias_act_kernel<1, int64_t><<<grid_for(work), 256, 0, s>>>(y, rows, cols, ld, bias, relu);
  return done(cudaGetLastError());
}

gemm_status_t kselect_maxpool2x2(const float* x, int32_t N, int32_t H, int32_t W, int32_t C, float* out,
                                 void* stream) {
  if (N < 0 || H < 0 || W < 0 || C < 1 || (H % 2) || (W % 2)) return GEMM_ERR_INVALID_ARG;
  const int64_t total = (int64_t)N * (H / 2) * (W / 2) * C;
  if (total == 0) return GEMM_OK;
  if (!x || !out) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = C % 4 == 0 && aligned16(x) && aligned16(out);
  const int64_t work = vec ? total / 4 : total;
  const bool small = work < ((int64_t)1 << 31) - 152LL * 32 * 256;
  if (vec && small) maxpool2x2_kernel<4, int32_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out);
  else if (vec) maxpool2x2_kernel<4, int64_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out);
  else if (small) maxpool2x2_kernel<1, int32_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out);
  else maxpool2x2_kernel<1, int64_t><<<grid_for(work), 256, 0, s>>>(x, N, H, W, C, out);
  return done(cudaGetLastError());
}

gemm_status_t kselect_im2col3x3_nchw(const float* x, int32_t N, int32_t C, int32_t H, int32_t W, float* out,
                                     int64_t ld, void* stream) {
  if (N < 0 || H < 0 || W < 0 || C < 1 || ld < 9LL * C) return GEMM_ERR_INVALID_ARG;
  const int64_t total = (int64_t)N * H * W * 9 * C;
  if (total == 0) return GEMM_OK;
  if (!x || !out) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (total < ((int64_t)1 << 31) - 152LL * 32 * 256)
    im2col3x3_nchw_kernel<int32_t><<<grid_for(total), 256, 0, s>>>(x, N, C, H, W, out, ld);
  else
    im2col3x3_nchw_kernel<int64_t><<<grid_for(total), 256, 0, s>>>(x, N, C, H, W, out, ld);
  return done(cudaGetLastError());
}

gemm_status_t kselect_bias_act_nchw(float* y, int32_t N, int32_t C, int64_t HW, const float* bias, int32_t relu,
                                    void* stream) {
  if (N < 0 || C < 1 || HW < 0) return GEMM_ERR_INVALID_ARG;
  const int64_t total = (int64_t)N * C * HW;
  if (total == 0) return GEMM_OK;
  if (!y) return GEMM_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (total < ((int64_t)1 << 31) - 152LL * 32 * 256)
    bias_act_nchw_kernel<int32_t><<<grid_for(total), 256, 0, s>>>(y, N, C, HW, bias, relu);
  else
    bias_act_nchw_kernel<int64_t><<<grid_for(total), 256, 0, s>>>(y, N, C, HW, bias, relu);
  return done(cudaGetLastError());
}

}  // extern "C"
