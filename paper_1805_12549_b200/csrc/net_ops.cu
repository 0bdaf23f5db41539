// The ungated operators of a channel-gated ResNet-18 (cgnet.h): patch matrix of the stem,
// pixel subsampling for the 1x1 stride-2 shortcuts, max pooling, global average pooling.
// NHWC bf16; each is one memory-bound kernel that moves 16-byte vectors where the channel
// count allows.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cgnet.h"
#include "common.cuh"
#include "ptx.cuh"

namespace {

constexpr int kBlock = 256;

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline int grid_for(long long items, int cap = 148 * 16) {
  long long g = (items + kBlock - 1) / kBlock;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

// Every operator is a dependent launch: its blocks are scheduled while the kernel in front ends, and wait here for it.
// (Its input is then not read-only for the kernel's whole life: it must not go through the non-coherent load path, so no
// __ldg and no __restrict__ on it.)
__device__ __forceinline__ void dependent_start() {
  cg::ptx::grid_launch_dependents();
  cg::ptx::grid_dependency_wait();
}

// One thread per group of eight consecutive columns of the patch matrix.
__global__ void __launch_bounds__(kBlock) im2col_kernel(const __nv_bfloat16* x,
                                                        __nv_bfloat16* __restrict__ a, int n, int h, int w,
                                                        int c, int k, int stride, int pad, int ho, int wo,
                                                        int k_pad) {
  dependent_start();
  const int vecs = k_pad >> 3;
  const long long total = (long long)n * ho * wo * vecs;
  const int kkc = k * k * c;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i % vecs);
    long long m = i / vecs;
    const int j = (int)(m % wo); m /= wo;
    const int ii = (int)(m % ho);
    const int img = (int)(m / ho);
    __align__(16) __nv_bfloat16 out[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int col = v * 8 + e;
      __nv_bfloat16 val = __float2bfloat16(0.f);
      if (col < kkc) {
        const int ci = col % c, rs = col / c, s = rs % k, r = rs / k;
        const int yy = ii * stride + r - pad, xx = j * stride + s - pad;
        if (yy >= 0 && yy < h && xx >= 0 && xx < w) val = x[(((long long)img * h + yy) * w + xx) * c + ci];
      }
      out[e] = val;
    }
    *reinterpret_cast<uint4*>(a + i * 8) = *reinterpret_cast<const uint4*>(out);
  }
}

// The same for compile-time filter size, channel count and stride (the divisions become
// multiplications), one block per output row: the k input rows the output row reads are staged
// in shared memory once, then every thread gathers 16-byte vectors of the patch matrix from it.
template <int K, int C, int STRIDE>
__global__ void __launch_bounds__(kBlock) im2col_rows_kernel(const __nv_bfloat16* x,
                                                             __nv_bfloat16* __restrict__ a, int n, int h, int w,
                                                             int pad, int ho, int wo, int k_pad) {
  extern __shared__ __nv_bfloat16 rows[];               // [K][(w + 2*pad) * C], zero where outside the image
  dependent_start();
  const int row_len = (w + 2 * pad) * C;
  const int vecs = k_pad >> 3;
  constexpr int kkc = K * K * C;
  for (int job = blockIdx.x; job < n * ho; job += gridDim.x) {
    const int img = job / ho, i = job - img * ho;
    __syncthreads();                                    // the previous row's readers are done
    for (int t = threadIdx.x; t < K * row_len; t += blockDim.x) {
      const int r = t / row_len, q = t - r * row_len;
      const int yy = i * STRIDE + r - pad, xx = q / C - pad;
      __nv_bfloat16 v = __float2bfloat16(0.f);
      if (yy >= 0 && yy < h && xx >= 0 && xx < w) v = x[(((long long)img * h + yy) * w + xx) * C + (q % C)];
      rows[t] = v;
    }
    __syncthreads();
    __nv_bfloat16* out_row = a + (long long)job * wo * k_pad;
    for (int t = threadIdx.x; t < wo * vecs; t += blockDim.x) {
      const int j = t / vecs, v = t - j * vecs;
      __align__(16) __nv_bfloat16 out[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int col = v * 8 + e;
        // column (r, s, ci) reads the staged row r at pixel j*STRIDE + s (padding included), channel ci
        const int r = col / (K * C), sc = col - r * (K * C);
        out[e] = col < kkc ? rows[r * row_len + j * STRIDE * C + sc] : __float2bfloat16(0.f);
      }
      *reinterpret_cast<uint4*>(out_row + (long long)t * 8) = *reinterpret_cast<const uint4*>(out);
    }
  }
}

__global__ void __launch_bounds__(kBlock) subsample_kernel(const uint4* x, uint4* __restrict__ y,
                                                           int n, int h, int w, int cv, int stride, int ho,
                                                           int wo) {
  dependent_start();
  const long long total = (long long)n * ho * wo * cv;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i % cv);
    long long m = i / cv;
    const int j = (int)(m % wo); m /= wo;
    const int ii = (int)(m % ho);
    const int img = (int)(m / ho);
    y[i] = x[(((long long)img * h + ii * stride) * w + j * stride) * cv + v];
  }
}

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a),
                                   *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}

__global__ void __launch_bounds__(kBlock) maxpool_kernel(const uint4* x, uint4* __restrict__ y,
                                                         int n, int h, int w, int cv, int k, int stride, int pad,
                                                         int ho, int wo) {
  dependent_start();
  const long long total = (long long)n * ho * wo * cv;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i % cv);
    long long m = i / cv;
    const int j = (int)(m % wo); m /= wo;
    const int ii = (int)(m % ho);
    const int img = (int)(m / ho);
    const uint32_t ninf = 0xff80ff80u;   // two bf16 -inf
    uint4 best = make_uint4(ninf, ninf, ninf, ninf);
    for (int r = 0; r < k; ++r) {
      const int yy = ii * stride + r - pad;
      if (yy < 0 || yy >= h) continue;
      for (int s = 0; s < k; ++s) {
        const int xx = j * stride + s - pad;
        if (xx < 0 || xx >= w) continue;
        const uint4 t = x[(((long long)img * h + yy) * w + xx) * cv + v];
        best.x = max_bf16x2(best.x, t.x); best.y = max_bf16x2(best.y, t.y);
        best.z = max_bf16x2(best.z, t.z); best.w = max_bf16x2(best.w, t.w);
      }
    }
    y[i] = best;
  }
}

// The 3x3, stride-2, padding-1 pooling of a ResNet, for up to 2^31 outputs: one output vector per thread, its
// nine loads in flight together, indices by multiplications.  The general kernel spent its time on 64-bit divisions
// and one load after the other: 128 x 112x112 x 64 (256 MB) 73 us, here 42.
__global__ void __launch_bounds__(kBlock) maxpool3_kernel(const uint4* x, uint4* __restrict__ y, unsigned total,
                                                          int h, int w, int cv, int ho, int wo, cg::FastDiv div_cv,
                                                          cg::FastDiv div_wo, cg::FastDiv div_ho) {
  dependent_start();
  const unsigned i = blockIdx.x * kBlock + threadIdx.x;
  if (i >= total) return;
  const unsigned m = div_cv.div(i), v = i - m * (unsigned)cv;
  const unsigned row = div_wo.div(m), j = m - row * (unsigned)wo;
  const unsigned img = div_ho.div(row), ii = row - img * (unsigned)ho;
  const uint32_t ninf = 0xff80ff80u;   // two bf16 -inf
  uint4 t[9];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int s = 0; s < 3; ++s) {
      const int yy = (int)ii * 2 + r - 1, xx = (int)j * 2 + s - 1;
      t[r * 3 + s] = make_uint4(ninf, ninf, ninf, ninf);
      if (yy >= 0 && yy < h && xx >= 0 && xx < w) t[r * 3 + s] = x[(((long long)img * h + yy) * w + xx) * cv + v];
    }
  uint4 best = t[0];
#pragma unroll
  for (int k = 1; k < 9; ++k) {
    best.x = max_bf16x2(best.x, t[k].x); best.y = max_bf16x2(best.y, t[k].y);
    best.z = max_bf16x2(best.z, t[k].z); best.w = max_bf16x2(best.w, t[k].w);
  }
  // (a window of NaN gives -inf, as with the general kernel's initial value)
  best.x = max_bf16x2(best.x, ninf); best.y = max_bf16x2(best.y, ninf);
  best.z = max_bf16x2(best.z, ninf); best.w = max_bf16x2(best.w, ninf);
  y[i] = best;
}

// One thread per (image, group of eight channels): fp32 sums over the pixels in order.  Where the threads do not fill the SMs,
// eight pixels' loads are in flight (with one or two, the 49 pixels of a 7x7 image are a chain of L2 reads) and a block has 64
// threads, which reach more SMs; else a load at a time, whose few registers let all the threads there be bring as much.  us of
// the former / the latter: 7x7 x 512, 128 images 5.9 / 8.3, 4096 images 34 / 41; 7x7 x 2048, 4096 images 155 / 121; 65536 pixels
// x 512 52 / 27.
template <int kBlockThreads, int kLoads>
__global__ void __launch_bounds__(kBlockThreads) avgpool_kernel(const uint4* x, uint4* __restrict__ y, int n, int hw, int cv) {
  dependent_start();
  const int total = n * cv;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int v = i % cv, img = i / cv;
    const uint4* src = x + (long long)img * hw * cv + v;
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    const unsigned pixels = (unsigned)hw;                        // (p runs up to seven past them)
    for (unsigned p = 0; p < pixels; p += kLoads) {
      uint4 t[kLoads];
#pragma unroll
      for (int k = 0; k < kLoads; ++k) t[k] = p + k < pixels ? src[(long long)(p + k) * cv] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int k = 0; k < kLoads; ++k) {
        if (p + k >= pixels) break;
        const __nv_bfloat16* tb = reinterpret_cast<const __nv_bfloat16*>(&t[k]);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += __bfloat162float(tb[e]);
      }
    }
    __align__(16) __nv_bfloat16 out[8];
    const float inv = 1.0f / (float)hw;
#pragma unroll
    for (int e = 0; e < 8; ++e) out[e] = __float2bfloat16_rn(acc[e] * inv);
    y[i] = *reinterpret_cast<const uint4*>(out);
  }
}

template <typename... Args>
cg_status launch(void (*kernel)(Args...), unsigned blocks, int threads, size_t smem, void* stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = static_cast<cudaStream_t>(stream);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? CG_OK : CG_ERR_CUDA;
}

}  // namespace

extern "C" {

cg_status cg_im2col_bf16(const void* x, void* a, int n, int h, int w, int c, int k, int stride, int pad,
                         int k_pad, void* cuda_stream) {
  if (!x || !a || n <= 0 || h <= 0 || w <= 0 || c <= 0 || k <= 0 || stride <= 0 || pad < 0) return CG_ERR_INVALID_ARG;
  if (k_pad < k * k * c || (k_pad & 7) || h + 2 * pad < k || w + 2 * pad < k) return CG_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(a)) return CG_ERR_ALIGNMENT;
  const int ho = (h + 2 * pad - k) / stride + 1, wo = (w + 2 * pad - k) / stride + 1;
  const long long items = (long long)n * ho * wo * (k_pad >> 3);
  const size_t stage = (size_t)k * (w + 2 * pad) * c * sizeof(__nv_bfloat16);
  if (k == 7 && c == 3 && stride == 2 && stage <= 48 * 1024) {   // the ResNet stem
    const int blocks = n * ho < 148 * 8 ? n * ho : 148 * 8;
    return launch(im2col_rows_kernel<7, 3, 2>, (unsigned)blocks, kBlock, stage, cuda_stream,
                  static_cast<const __nv_bfloat16*>(x), static_cast<__nv_bfloat16*>(a), n, h, w, pad, ho, wo, k_pad);
  }
  return launch(im2col_kernel, (unsigned)grid_for(items), kBlock, 0, cuda_stream, static_cast<const __nv_bfloat16*>(x),
                static_cast<__nv_bfloat16*>(a), n, h, w, c, k, stride, pad, ho, wo, k_pad);
}

cg_status cg_subsample_bf16(const void* x, void* y, int n, int h, int w, int c, int stride, void* cuda_stream) {
  if (!x || !y || n <= 0 || h <= 0 || w <= 0 || c <= 0 || stride <= 0 || (c & 7)) return CG_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(y)) return CG_ERR_ALIGNMENT;
  const int ho = (h + stride - 1) / stride, wo = (w + stride - 1) / stride;
  const long long items = (long long)n * ho * wo * (c >> 3);
  return launch(subsample_kernel, (unsigned)grid_for(items), kBlock, 0, cuda_stream, static_cast<const uint4*>(x),
                static_cast<uint4*>(y), n, h, w, c >> 3, stride, ho, wo);
}

cg_status cg_maxpool_bf16(const void* x, void* y, int n, int h, int w, int c, int k, int stride, int pad,
                          void* cuda_stream) {
  if (!x || !y || n <= 0 || h <= 0 || w <= 0 || c <= 0 || k <= 0 || stride <= 0 || pad < 0 || (c & 7)) return CG_ERR_INVALID_ARG;
  if (pad >= k || h + 2 * pad < k || w + 2 * pad < k) return CG_ERR_INVALID_ARG;   // every window holds a pixel
  if (!aligned16(x) || !aligned16(y)) return CG_ERR_ALIGNMENT;
  const int ho = (h + 2 * pad - k) / stride + 1, wo = (w + 2 * pad - k) / stride + 1;
  const long long items = (long long)n * ho * wo * (c >> 3);
  if (k == 3 && stride == 2 && pad == 1 && items < (1ll << 31) - kBlock) {
    cg::FastDiv div_cv, div_wo, div_ho;
    div_cv.set((uint32_t)(c >> 3)); div_wo.set((uint32_t)wo); div_ho.set((uint32_t)ho);
    return launch(maxpool3_kernel, (unsigned)((items + kBlock - 1) / kBlock), kBlock, 0, cuda_stream, static_cast<const uint4*>(x),
                  static_cast<uint4*>(y), (unsigned)items, h, w, c >> 3, ho, wo, div_cv, div_wo, div_ho);
  }
  return launch(maxpool_kernel, (unsigned)grid_for(items), kBlock, 0, cuda_stream, static_cast<const uint4*>(x),
                static_cast<uint4*>(y), n, h, w, c >> 3, k, stride, pad, ho, wo);
}

cg_status cg_avgpool_bf16(const void* x, void* y, int n, int hw, int c, void* cuda_stream) {
  if (!x || !y || n <= 0 || hw <= 0 || c <= 0 || (c & 7)) return CG_ERR_INVALID_ARG;
  if (!aligned16(x) || !aligned16(y)) return CG_ERR_ALIGNMENT;
  const long long threads = (long long)n * (c >> 3);
  if (threads > 148 * 2048)
    return launch(avgpool_kernel<kBlock, 1>, (unsigned)grid_for(threads), kBlock, 0, cuda_stream, static_cast<const uint4*>(x),
                  static_cast<uint4*>(y), n, hw, c >> 3);
  return launch(avgpool_kernel<64, 8>, (unsigned)((threads + 63) / 64), 64, 0, cuda_stream, static_cast<const uint4*>(x),
                static_cast<uint4*>(y), n, hw, c >> 3);
}

}  // extern "C"
