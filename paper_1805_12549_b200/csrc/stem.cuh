// The 7x7 stride-2 stem convolution of a ResNet straight from the image (stem.cu).
#pragma once

#include "common.cuh"

namespace cg {

constexpr size_t kStemWeightBytes = 3 * 64 * 128;   // the filter as the kernel's shared memory holds it

// x [n,h,w,3] bf16; w_base [64][k_pad], columns (r*7 + s)*3 + c; y [n,ho,wo,64]; ws: kStemWeightBytes.
// Two launches: the filter into ws, then the convolution with its batch norm, gate and activation.
int launch_stem(const void* x, int n, int h, int w, const void* w_base, int k_pad, const cg_bn_params& bn,
                const float* delta, float eps, int relu, void* y, void* ws, unsigned long long* counters,
                cudaStream_t stream);

// How launch_stem_pool cuts n images into strips: worked out by its first call for these extents, kept by the handle.
struct StemPoolPlan {
  int n, h, w;             // 0: none yet
  int sms, segs, per;      // a column of an image in `segs` strips of `per` pooled rows
};
// The stem and the 3x3 stride-2 max pooling behind it in one launch (stem_pool.cu): y as above, pooled [n,hp,wp,64].
// Even image widths only, extents up to kStemPoolMaxExtent (words of an image row are counted in 32 bits).
constexpr int kStemPoolMaxExtent = 1 << 30;
int launch_stem_pool(StemPoolPlan* plan, const void* x, int n, int h, int w, const void* w_base, int k_pad, const cg_bn_params& bn,
                     const float* delta, float eps, int relu, void* y, void* pooled, unsigned long long* counters,
                     cudaStream_t stream);
// Whether that is faster than launch_stem and a pooling kernel.
bool stem_pool_pays(int n, int h, int w);

}  // namespace cg
