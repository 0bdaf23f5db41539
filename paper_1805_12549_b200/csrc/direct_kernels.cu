// CUDA-core direct convolution of the channel-gated layer: the path for fp32 layers and for
// every shape the tensor-core path does not take.
//
// One warp owns one (pixel row m, 32-channel block q): lane = output channel.  Each lane runs
// the base-path sum (Section 3.1), takes the gate decision (Eq. 2/3), runs the conditional-path
// sum only if its own gate fired (Eq. 1), applies the path's batch norm and ReLU, and the
// warp's ballot is the mask word.  Floating-point sums run in the order (r, s, c_in) with
// separately rounded multiply and add, so results do not depend on the launch shape.
#include <algorithm>
#include <cstring>

#include "common.cuh"
#include "direct_point.cuh"
#include "ptx.cuh"

namespace cg {
namespace {

__device__ __forceinline__ int conv_point_i8(const LayerDims& L, const int8_t* __restrict__ x,
                                             const int8_t* __restrict__ w, int n, int ho, int wo,
                                             int co, int c_lo, int cw) {
  int acc = 0;
  for (int r = 0; r < L.kh; ++r) {
    const int hi = ho * L.stride + r - L.pad;
    if (hi < 0 || hi >= L.h) continue;
    for (int s = 0; s < L.kw; ++s) {
      const int wi = wo * L.stride + s - L.pad;
      if (wi < 0 || wi >= L.w) continue;
      const int8_t* xp = x + (((long long)n * L.h + hi) * L.w + wi) * L.c_in + c_lo;
      const int8_t* wp = w + (((long long)co * L.kh + r) * L.kw + s) * cw;
      int ci = 0;
      // four products per instruction where both runs are 4-byte aligned (integer sums do not
      // depend on the order)
      if ((((uintptr_t)xp | (uintptr_t)wp) & 3u) == 0)
        for (; ci + 4 <= cw; ci += 4) acc = __dp4a(*(const int*)(xp + ci), *(const int*)(wp + ci), acc);
      for (; ci < cw; ++ci) acc += (int)xp[ci] * (int)wp[ci];
    }
  }
  return acc;
}

// Channel grouping (Section 3.3): the conditional path of output group g reads every input
// channel outside [g*c_p, (g+1)*c_p), in ascending order; weights are [c_out][kh][kw][c_r].
template <typename T>
__device__ __forceinline__ float conv_point_others(const LayerDims& L, const T* __restrict__ x,
                                                   const T* __restrict__ w, int n, int ho, int wo,
                                                   int co, int g) {
  float acc = 0.f;
  const int lo = g * L.c_p, hi2 = lo + L.c_p;
  for (int r = 0; r < L.kh; ++r) {
    const int hi = ho * L.stride + r - L.pad;
    if (hi < 0 || hi >= L.h) continue;
    for (int s = 0; s < L.kw; ++s) {
      const int wi = wo * L.stride + s - L.pad;
      if (wi < 0 || wi >= L.w) continue;
      const T* xp = x + (((long long)n * L.h + hi) * L.w + wi) * L.c_in;
      const T* wp = w + (((long long)co * L.kh + r) * L.kw + s) * L.c_r;
      for (int ci = 0; ci < lo; ++ci)
        acc = __fadd_rn(acc, __fmul_rn(Elem<T>::ld(xp + ci), Elem<T>::ld(wp + ci)));
      for (int ci = hi2; ci < L.c_in; ++ci)
        acc = __fadd_rn(acc, __fmul_rn(Elem<T>::ld(xp + ci), Elem<T>::ld(wp + ci - L.c_p)));
    }
  }
  return acc;
}

__device__ __forceinline__ int conv_point_others_i8(const LayerDims& L, const int8_t* __restrict__ x,
                                                    const int8_t* __restrict__ w, int n, int ho,
                                                    int wo, int co, int g) {
  int acc = 0;
  const int lo = g * L.c_p, hi2 = lo + L.c_p;
  for (int r = 0; r < L.kh; ++r) {
    const int hi = ho * L.stride + r - L.pad;
    if (hi < 0 || hi >= L.h) continue;
    for (int s = 0; s < L.kw; ++s) {
      const int wi = wo * L.stride + s - L.pad;
      if (wi < 0 || wi >= L.w) continue;
      const int8_t* xp = x + (((long long)n * L.h + hi) * L.w + wi) * L.c_in;
      const int8_t* wp = w + (((long long)co * L.kh + r) * L.kw + s) * L.c_r;
      for (int ci = 0; ci < lo; ++ci) acc += (int)xp[ci] * (int)wp[ci];
      for (int ci = hi2; ci < L.c_in; ++ci) acc += (int)xp[ci] * (int)wp[ci - L.c_p];
    }
  }
  return acc;
}

constexpr int kThreads = 256;

template <typename TIn, typename TOut>
__global__ void __launch_bounds__(kThreads)
direct_gated_conv_kernel(LayerDims L, const TIn* __restrict__ x, const TIn* __restrict__ w_base,
                         const TIn* __restrict__ w_cond, cg_bn_params bn,
                         const float* __restrict__ delta, const TOut* __restrict__ residual,
                         TOut* __restrict__ y, uint32_t* __restrict__ mask,
                         float* __restrict__ p_out, int base_only,
                         unsigned long long* __restrict__ counters,
                         int chan_pass = 0, int* __restrict__ chan_cnt = nullptr, float chan_need = 0.f) {
  // chan_pass (channel-wise gate, Eq. 4): 1 = first pass: partial sums to p_out and, per image
  // and output channel, the number of firing gates to chan_cnt; 2 = second pass: partial sums
  // read back from p_out, conditional path only where the activation's gate fires AND the
  // channel's count reaches chan_need = tau_c * h' * w'.
  extern __shared__ float s_consts[];   // 6 * c_out: t, a1, b1, a2, b2, t2
  __shared__ unsigned long long s_active;
  float* s_t = s_consts;
  float* s_a1 = s_t + L.c_out;
  float* s_b1 = s_a1 + L.c_out;
  float* s_a2 = s_b1 + L.c_out;
  float* s_b2 = s_a2 + L.c_out;
  float* s_t2 = s_b2 + L.c_out;
  if (threadIdx.x == 0) s_active = 0ull;
  if (!base_only) {
    for (int c = threadIdx.x; c < L.c_out; c += blockDim.x) {
      const ChannelConsts k = fold_channel(bn, delta, L.eps, c);
      s_t[c] = k.t; s_a1[c] = k.a1; s_b1[c] = k.b1; s_a2[c] = k.a2; s_b2[c] = k.b2; s_t2[c] = k.t2;
    }
  }
  __syncthreads();

  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long warp0 = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long items = L.m * L.words;
  unsigned long long my_active = 0;
  for (long long it = warp0; it < items; it += warps) {
    const long long m = it / L.words;
    const int q = (int)(it - m * L.words);
    const int co = q * 32 + lane;
    const bool valid = co < L.c_out;
    const int wo = (int)(m % L.wo);
    const int ho = (int)((m / L.wo) % L.ho);
    const int n = (int)(m / ((long long)L.wo * L.ho));
    bool fire = false;
    if (valid) {
      const int grp = L.grouping ? co / (L.c_out / L.groups) : 0;   // input group of the base path
      const float p = chan_pass == 2 ? p_out[m * L.c_out + co]
                                     : conv_point<TIn>(L, x, w_base, n, ho, wo, co, grp * L.c_p, L.c_p);
      if (base_only) {
        p_out[m * L.c_out + co] = p;
      } else if (chan_pass == 1) {
        p_out[m * L.c_out + co] = p;
        if (p >= s_t[co] && p <= s_t2[co]) atomicAdd(&chan_cnt[(long long)n * L.c_out + co], 1);
      } else {
        fire = (p >= s_t[co]) && (p <= s_t2[co]);   // NaN compares false; t2 = +inf unless the gate is two-sided
        if (chan_pass == 2) {
          const bool on = ((float)chan_cnt[(long long)n * L.c_out + co] >= chan_need);
          fire = fire && on;
          if (!on && ho == 0 && wo == 0) atomicAdd(&counters[CNT_CH_SKIPPED], 1ull);
        }
        float v;
        if (fire) {
          const float r = L.grouping ? conv_point_others<TIn>(L, x, w_cond, n, ho, wo, co, grp)
                                     : conv_point<TIn>(L, x, w_cond, n, ho, wo, co, L.c_p, L.c_r);
          v = __fadd_rn(__fmul_rn(s_a2[co], __fadd_rn(p, r)), s_b2[co]);
        } else {
          v = __fadd_rn(__fmul_rn(s_a1[co], p), s_b1[co]);
        }
        if (residual) v = __fadd_rn(v, (float)residual[m * L.c_out + co]);
        if (L.relu) v = (v > 0.f) ? v : 0.f;
        st_out(y + m * L.c_out + co, v);
      }
    }
    if (!base_only && chan_pass != 1) {
      const unsigned word = __ballot_sync(0xffffffffu, fire);
      if (lane == 0) {
        if (mask) mask[it] = word;
        my_active += __popc(word);
      }
    }
  }
  if (!base_only && chan_pass != 1) {
    if (lane == 0 && my_active) atomicAdd(&s_active, my_active);
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(&counters[CNT_CALLS], 1ull);
    if (threadIdx.x == 0 && s_active) {
      atomicAdd(&counters[CNT_ACTIVE], s_active);
    }
  }
}

__global__ void __launch_bounds__(kThreads)
direct_gated_conv_i8_kernel(LayerDims L, const int8_t* __restrict__ x,
                            const int8_t* __restrict__ w_base, const int8_t* __restrict__ w_cond,
                            cg_bn_params bn, int8_t* __restrict__ y, uint32_t* __restrict__ mask,
                            int* __restrict__ p_out, int base_only,
                            unsigned long long* __restrict__ counters) {
  __shared__ unsigned long long s_active;
  if (threadIdx.x == 0) s_active = 0ull;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  const long long warp0 = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long items = L.m * L.words;
  unsigned long long my_active = 0;
  for (long long it = warp0; it < items; it += warps) {
    const long long m = it / L.words;
    const int q = (int)(it - m * L.words);
    const int co = q * 32 + lane;
    const bool valid = co < L.c_out;
    const int wo = (int)(m % L.wo);
    const int ho = (int)((m / L.wo) % L.ho);
    const int n = (int)(m / ((long long)L.wo * L.ho));
    bool fire = false;
    if (valid) {
      const int grp = L.grouping ? co / (L.c_out / L.groups) : 0;
      const int p = conv_point_i8(L, x, w_base, n, ho, wo, co, grp * L.c_p, L.c_p);
      if (base_only) {
        p_out[m * L.c_out + co] = p;
      } else {
        fire = (p >= bn.q_gate_thr[co]);
        long long acc = p;
        if (fire) acc += L.grouping ? conv_point_others_i8(L, x, w_cond, n, ho, wo, co, grp)
                                    : conv_point_i8(L, x, w_cond, n, ho, wo, co, L.c_p, L.c_r);
        const bool full = fire;
        const long long mul = full ? bn.q_mul_full[co] : bn.q_mul_base[co];
        const long long off = full ? bn.q_off_full[co] : bn.q_off_base[co];
        long long qv = (acc * mul + off + (1ll << (L.shift - 1))) >> L.shift;
        const long long lo = L.relu ? 0 : -128;
        qv = qv < lo ? lo : (qv > 127 ? 127 : qv);
        y[m * L.c_out + co] = (int8_t)qv;
      }
    }
    if (!base_only) {
      const unsigned word = __ballot_sync(0xffffffffu, fire);
      if (lane == 0) {
        if (mask) mask[it] = word;
        my_active += __popc(word);
      }
    }
  }
  if (!base_only) {
    if (lane == 0 && my_active) atomicAdd(&s_active, my_active);
    __syncthreads();
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(&counters[CNT_CALLS], 1ull);
    if (threadIdx.x == 0 && s_active) {
      atomicAdd(&counters[CNT_ACTIVE], s_active);
    }
  }
}

// ---- the tiled direct kernel ---------------------------------------------------------------------------
// The same sums in the same order -- (r, s, c_in), one accumulator per output and path, taps outside the image
// left out -- from operands staged in shared memory: a block owns TM pixels x TC channels, a thread PXT pixels
// x CH channels.  A run of kStage K elements (tap-major, then channel) is gathered per stage: four consecutive
// channels of a tap per load, converted to fp32, two stages in flight.  The warp-per-output kernel above waits
// for one pair of global loads per product: 156 us for the partial sums of four images of 56x56 (64 channels,
// c_p = 16), here 19.2; counters there: shared-memory reads 58 % of their rate, issue slots 48 %, DRAM 1 %.  It remains for channel counts that are not multiples of four, channel
// grouping and the channel-wise gate.
// Products and sums are rounded separately, for bf16 operands too: their products are exact in fp32 only inside its
// normal range, so a fused multiply-add is another sum where one is below 2^-126 or beyond 2^128.

// The filter rows [r0, r0 + kh) and columns [s0, s0 + kw) that some output pixel meets inside the image; the others
// meet padding only, and are not run through.  (All of them unless the image is smaller than the filter's reach: a
// 3x3 layer on one pixel has one tap, 128 channels 23.2 us with all nine run through, 7x7 on 2x2 images 9 of 49.)
struct TapBox {
  int r0, s0, kh, kw;
};
TapBox tap_box(const LayerDims& L) {
  auto first = [&](int out) { return (int)std::max(0ll, L.pad - (out - 1ll) * L.stride); };
  auto end = [&](int k, int in) { return (int)std::min((long long)k, (long long)L.pad + in); };
  TapBox b = {first(L.ho), first(L.wo), 0, 0};
  b.kh = std::max(0, end(L.kh, L.h) - b.r0); b.kw = std::max(0, end(L.kw, L.w) - b.s0);   // (0: every sum is empty)
  return b;
}

// Four channels as they lie in memory; they become fp32 on their way to shared memory.
template <typename T> struct Four { using Raw = float4; };
template <> struct Four<__nv_bfloat16> { using Raw = uint2; };
__device__ __forceinline__ float4 widen(float4 v) { return v; }
__device__ __forceinline__ float4 widen(uint2 v) {
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                     __uint_as_float(v.y & 0xffff0000u));
}
// Pixels by ordinary loads, and no __restrict__ on what they read: the kernel in front, whose end this one's launch does not
// wait for, may still be writing them.  Weights by the read-only path.  (us with all loads on the read-only path / this, with the
// loads of a stage in front of the barrier and widened behind it: 16 channels of 8x8, two images, fp32 5.1 / 5.1 in a chain; 64
// channels of 28x28, 64 images, fp32 240 / 231; partial sums of four images of 28x28 x 128 33.8 / 32.0, of 56x56 x 64 18.3 / 18.9.)
// Inline loads that the compiler may move are no way out: it may also move them out of the test that keeps them in bounds.
template <bool READ_ONLY, typename T> __device__ __forceinline__ typename Four<T>::Raw load4(const T* p) {
  const typename Four<T>::Raw* q = reinterpret_cast<const typename Four<T>::Raw*>(p);
  return READ_ONLY ? __ldg(q) : *q;
}
__device__ __forceinline__ float mul_add(float a, float b, float c) { return __fadd_rn(c, __fmul_rn(a, b)); }

template <int NTH, int TC, int PXT, int CH>
struct DirectTile {
  static constexpr int kGroups = TC / CH;                  // threads per pixel
  static constexpr int kPixGroups = NTH / kGroups;
  static constexpr int TM = kPixGroups * PXT;
  // K elements per stage: 32, or 128 where a block has little to compute and waits for its loads instead
  static constexpr int kStage = PXT == 1 ? 128 : 32;
  static constexpr int kXPitch = kStage + 4;
  // weights: [K][channel] where a thread takes four channels, [channel][K] where it takes one
  static constexpr int kWPitch = CH == 4 ? TC + 4 : kStage + 4, kWSize = CH == 4 ? kStage * kWPitch : TC * kWPitch;
  struct Buffers {
    float x[2][TM * kXPitch];
    float w[2][kWSize];
    uint8_t ok[2][kStage / 4 * TM];
  };
};

// BOX: the taps of tap_box() only (an instance of its own: the index arithmetic of its weights costs the others 4 %)
template <typename T, int NTH, int TC, int PXT, int CH, bool BOX>
__global__ void __launch_bounds__(NTH, PXT == 4 ? 2 : 3)
direct_tile_kernel(LayerDims L, const T* x, const T* __restrict__ w_base, const T* __restrict__ w_cond,
                   cg_bn_params bn, const float* __restrict__ delta, const T* residual, T* __restrict__ y,
                   uint32_t* __restrict__ mask, float* __restrict__ p_out, int base_only,
                   unsigned long long* __restrict__ counters, FastDiv div_base, FastDiv div_cond, FastDiv div_kw, TapBox box, uint64_t minus_zero) {
  using D = DirectTile<NTH, TC, PXT, CH>;
  constexpr int kStage = D::kStage;
  const TapBox taps = BOX ? box : TapBox{0, 0, L.kh, L.kw};
  ptx::grid_launch_dependents();
  extern __shared__ __align__(16) uint8_t dyn[];
  typename D::Buffers& S = *reinterpret_cast<typename D::Buffers*>(dyn);
  __shared__ float s_const[6][TC];
  __shared__ unsigned s_active;
  const int tid = threadIdx.x;
  const int cgi = tid % D::kGroups, pg = tid / D::kGroups;
  const int c0 = blockIdx.y * TC;
  const long long m0 = (long long)blockIdx.x * D::TM;
  if (tid == 0) s_active = 0;
  ptx::grid_dependency_wait();
  constexpr int kXTotal = D::TM * (kStage / 4), kWTotal = TC * (kStage / 4);   // loads of four channels per stage
  constexpr int kXUnits = (kXTotal + NTH - 1) / NTH, kWUnits = (kWTotal + NTH - 1) / NTH;
  // unit u = tid + NTH*i of a stage: pixel u % TM, K group u / TM.  TM divides NTH: a thread gathers one pixel.
  static_assert(NTH % D::TM == 0, "one pixel per thread");
  const int gx = tid % D::TM;
  int h0 = 0, w0 = 0;
  long long x_off = 0;                                     // element of the tap (0, 0) of the pixel
  const bool have_pixel = m0 + gx < L.m;
  if (have_pixel) {
    const unsigned m = (unsigned)(m0 + gx), hw = (unsigned)(L.ho * L.wo), n = m / hw, mi = m - n * hw, ho = mi / (unsigned)L.wo;
    h0 = (int)ho * L.stride - L.pad;
    w0 = (int)(mi - ho * (unsigned)L.wo) * L.stride - L.pad;
    x_off = (((long long)n * L.h + h0) * L.w + w0) * L.c_in;
  }
  typename Four<T>::Raw xr[kXUnits], wr[kWUnits];
  uint32_t okr = 0;

  // stage of the sums over `cw` channels from c_lo on: K elements [k0, k0 + kStage) into registers ...
  auto fetch = [&](const T* w, const FastDiv& div, int c_lo, int cw, int k0) {
    const int kt = taps.kh * taps.kw * cw, w_row = L.kh * L.kw * cw;
    okr = 0;
#pragma unroll
    for (int i = 0; i < kXUnits; ++i) {
      const int u = tid + NTH * i, k = k0 + u / D::TM * 4;
      xr[i] = {};
      if (have_pixel && u < kXTotal && k < kt) {
        const int tap = (int)div.div(k), ci = k - tap * cw, rr = (int)div_kw.div(tap), r = taps.r0 + rr, s = taps.s0 + tap - rr * taps.kw;
        if (h0 + r >= 0 && h0 + r < L.h && w0 + s >= 0 && w0 + s < L.w) {
          xr[i] = load4<false>(x + x_off + ((long long)r * L.w + s) * L.c_in + c_lo + ci);
          okr |= 1u << i;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kWUnits; ++i) {
      const int u = tid + NTH * i, c = u % TC, k = k0 + u / TC * 4;
      wr[i] = {};
      if (u < kWTotal && k < kt && c0 + c < L.c_out) {
        int at = k;                                        // element of the channel's filter
        if (BOX) {
          const int tap = (int)div.div(k), rr = (int)div_kw.div(tap);
          at = ((taps.r0 + rr) * L.kw + taps.s0 + tap - rr * taps.kw) * cw + k - tap * cw;
        }
        wr[i] = load4<true>(w + (long long)(c0 + c) * w_row + at);
      }
    }
  };
  // ... and from there to shared memory
  auto put = [&](int b) {
#pragma unroll
    for (int i = 0; i < kXUnits; ++i) {
      const int u = tid + NTH * i, g = u / D::TM;
      if (u >= kXTotal) break;
      *reinterpret_cast<float4*>(&S.x[b][gx * D::kXPitch + g * 4]) = widen(xr[i]);
      S.ok[b][g * D::TM + gx] = (uint8_t)((okr >> i) & 1u);
    }
#pragma unroll
    for (int i = 0; i < kWUnits; ++i) {
      const int u = tid + NTH * i, c = u % TC, g = u / TC;
      if (u >= kWTotal) break;
      const float4 v = widen(wr[i]);
      if (CH == 1) { *reinterpret_cast<float4*>(&S.w[b][c * D::kWPitch + g * 4]) = v; continue; }
      float* d = &S.w[b][g * 4 * D::kWPitch + c];
      d[0] = v.x; d[D::kWPitch] = v.y; d[2 * D::kWPitch] = v.z; d[3 * D::kWPitch] = v.w;
    }
  };
  int b = 0;                                               // buffer of the current stage
  // the sums, their first stage fetched already; `then` fetches what follows during the last stage
  auto sums = [&](float (&acc)[PXT][CH], const T* w, const FastDiv& div, int c_lo, int cw, auto then) {
#pragma unroll
    for (int i = 0; i < PXT; ++i)
#pragma unroll
      for (int e = 0; e < CH; ++e) acc[i][e] = 0.f;
    [[maybe_unused]] uint64_t a2[PXT][2];                    // CH = 4: the accumulators, two channels each
#pragma unroll
    for (int i = 0; i < PXT; ++i) a2[i][0] = a2[i][1] = 0;
    const int kt = taps.kh * taps.kw * cw, stages = (kt + kStage - 1) / kStage;
    // (the next loads are issued in front of the barrier: ordinary loads that come behind it in the program stay behind it)
    auto next = [&](int st) {
      if (st < stages) fetch(w, div, c_lo, cw, st * kStage);
      else if (st == stages) then();
    };
    put(b);
    next(1);
    __syncthreads();
    for (int st = 0; st < stages; ++st) {
      const int groups = min(kStage / 4, (kt - st * kStage) / 4);
      // operands of four K elements, read one group ahead where few warps share an SM
      float4 xv[2][PXT], wv[2][CH];                           // (of the weights: K elements x channels, or the reverse)
      bool ok[2][PXT];
      auto read = [&](int g, int h) {
#pragma unroll
        for (int i = 0; i < PXT; ++i) {
          const int px = pg + i * D::kPixGroups;
          xv[h][i] = *reinterpret_cast<const float4*>(&S.x[b][px * D::kXPitch + g * 4]);
          ok[h][i] = S.ok[b][g * D::TM + px] != 0;
        }
#pragma unroll
        for (int q = 0; q < CH; ++q)
          wv[h][q] = *reinterpret_cast<const float4*>(&S.w[b][CH == 1 ? cgi * D::kWPitch + g * 4 : (g * 4 + q) * D::kWPitch + cgi * 4]);
      };
      auto add = [&](int h) {
#pragma unroll
        for (int i = 0; i < PXT; ++i) {
          if (!ok[h][i]) continue;
          if constexpr (CH == 1) {
            acc[i][0] = mul_add(xv[h][i].x, wv[h][0].x, acc[i][0]); acc[i][0] = mul_add(xv[h][i].y, wv[h][0].y, acc[i][0]);
            acc[i][0] = mul_add(xv[h][i].z, wv[h][0].z, acc[i][0]); acc[i][0] = mul_add(xv[h][i].w, wv[h][0].w, acc[i][0]);
          } else {
            // Two channels per instruction, each rounded like the scalar operation.  The product is a*b + (-0), the
            // same in every case; -0 is a kernel argument, because of a product and a sum that it knows the compiler
            // makes one fused operation, .rn or not (its results differed from the definition's).
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float v = q == 0 ? xv[h][i].x : q == 1 ? xv[h][i].y : q == 2 ? xv[h][i].z : xv[h][i].w;
              const uint64_t vv = ptx::pack_f32x2(v, v);
              a2[i][0] = ptx::add_f32x2(a2[i][0], ptx::fma_f32x2(vv, ptx::pack_f32x2(wv[h][q].x, wv[h][q].y), minus_zero));
              a2[i][1] = ptx::add_f32x2(a2[i][1], ptx::fma_f32x2(vv, ptx::pack_f32x2(wv[h][q].z, wv[h][q].w), minus_zero));
            }
          }
        }
      };
      if (PXT > 1) {
#pragma unroll 2
        for (int g = 0; g < groups; ++g) { read(g, 0); add(0); }
      } else {
        read(0, 0);
      }
#pragma unroll 1
      for (int g = 0; PXT == 1 && g < groups; g += 2) {
        if (g + 1 < groups) read(g + 1, 1);
        add(0);
        if (g + 1 >= groups) break;
        if (g + 2 < groups) read(g + 2, 0);
        add(1);
      }
      b ^= 1;
      if (st + 1 < stages) { put(b); next(st + 2); }
      __syncthreads();
    }
    if constexpr (CH == 4) {
#pragma unroll
      for (int i = 0; i < PXT; ++i) {
        ptx::unpack_f32x2(a2[i][0], acc[i][0], acc[i][1]);
        ptx::unpack_f32x2(a2[i][1], acc[i][2], acc[i][3]);
      }
    }
  };

  float p[PXT][CH], rr[PXT][CH];
  const bool has_cond = !base_only && L.c_r > 0;
  fetch(w_base, div_base, 0, L.c_p, 0);
  if (!base_only && tid < TC && c0 + tid < L.c_out) {
    const ChannelConsts k = fold_channel(bn, delta, L.eps, c0 + tid);
    s_const[0][tid] = k.t; s_const[1][tid] = k.a1; s_const[2][tid] = k.b1;
    s_const[3][tid] = k.a2; s_const[4][tid] = k.b2; s_const[5][tid] = k.t2;
  }
  sums(p, w_base, div_base, 0, L.c_p, [&] { if (has_cond) fetch(w_cond, div_cond, L.c_p, L.c_r, 0); });
  const int cb = c0 + cgi * CH;
  if (base_only) {
#pragma unroll
    for (int i = 0; i < PXT; ++i) {
      const long long m = m0 + pg + i * D::kPixGroups;
      if (m >= L.m) continue;
#pragma unroll
      for (int e = 0; e < CH; ++e)
        if (cb + e < L.c_out) p_out[m * L.c_out + cb + e] = p[i][e];
    }
    return;
  }
  uint32_t fire[PXT];
  bool any = false;
#pragma unroll
  for (int i = 0; i < PXT; ++i) {
    fire[i] = 0;
    const long long m = m0 + pg + i * D::kPixGroups;
#pragma unroll
    for (int e = 0; e < CH; ++e) {
      const int c = cgi * CH + e;
      // (a NaN sum does not fire)
      if (m < L.m && cb + e < L.c_out && p[i][e] >= s_const[0][c] && p[i][e] <= s_const[5][c]) fire[i] |= 1u << e;
    }
    any = any || fire[i] != 0;
  }
#pragma unroll
  for (int i = 0; i < PXT; ++i)
#pragma unroll
    for (int e = 0; e < CH; ++e) rr[i][e] = 0.f;
  if (__syncthreads_or(any) && has_cond) sums(rr, w_cond, div_cond, L.c_p, L.c_r, [] {});
  unsigned active = 0;
#pragma unroll
  for (int i = 0; i < PXT; ++i) {
    const long long m = m0 + pg + i * D::kPixGroups;
    constexpr int kPerWord = 32 / CH, kWordLanes = D::kGroups < kPerWord ? D::kGroups : kPerWord;
    uint32_t word = fire[i] << (CH * (cgi % kPerWord));
#pragma unroll
    for (int o = 1; o < kWordLanes; o <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, o);
    if (m >= L.m) continue;
    if (cgi % kPerWord == 0 && cb < L.c_out) {
      active += __popc(word);
      if (mask && TC >= 32) mask[m * L.words + (cb >> 5)] = word;
      if (mask && TC == 16) {                              // half a word, and the empty half behind the last channels
        unsigned short* half = reinterpret_cast<unsigned short*>(mask) + m * L.words * 2 + (cb >> 4);
        half[0] = (unsigned short)word;
        if (cb + 16 >= L.c_out && !((cb >> 4) & 1)) half[1] = 0;
      }
    }
#pragma unroll
    for (int e = 0; e < CH; ++e) {
      const int c = cgi * CH + e;
      if (cb + e >= L.c_out) break;
      float v = (fire[i] >> e) & 1u ? __fadd_rn(__fmul_rn(s_const[3][c], __fadd_rn(p[i][e], rr[i][e])), s_const[4][c])
                                    : __fadd_rn(__fmul_rn(s_const[1][c], p[i][e]), s_const[2][c]);
      if (residual) v = __fadd_rn(v, (float)residual[m * L.c_out + cb + e]);
      if (L.relu) v = (v > 0.f) ? v : 0.f;
      st_out(y + m * L.c_out + cb + e, v);
    }
  }
  if (active) atomicAdd(&s_active, active);
  __syncthreads();
  if (tid == 0) {
    if (s_active) atomicAdd(&counters[CNT_ACTIVE], (unsigned long long)s_active);
    if (blockIdx.x == 0 && blockIdx.y == 0) atomicAdd(&counters[CNT_CALLS], 1ull);
  }
}

template <typename T, int NTH, int TC, int PXT, int CH, bool BOX = false>
int launch_tile(const LayerDims& L, const TapBox& taps, const void* x, const void* w_base, const void* w_cond, const cg_bn_params& bn,
                const float* delta, const void* residual, void* y, uint32_t* mask, void* p_out, int base_only,
                unsigned long long* counters, cudaStream_t stream) {
  using D = DirectTile<NTH, TC, PXT, CH>;
  const dim3 grid((unsigned)((L.m + D::TM - 1) / D::TM), (unsigned)((L.c_out + TC - 1) / TC), 1);
  const size_t smem = sizeof(typename D::Buffers);
  static bool set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  if (smem > 48 * 1024 && !set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(direct_tile_kernel<T, NTH, TC, PXT, CH, BOX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    set[dev] = true;
  }
  FastDiv div_base, div_cond, div_kw;
  div_base.set((uint32_t)L.c_p); div_cond.set((uint32_t)(L.c_r > 0 ? L.c_r : 1)); div_kw.set((uint32_t)std::max(1, BOX ? taps.kw : L.kw));
  // a programmatic dependent launch, like the tensor-core kernels
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid; cfg.blockDim = dim3(NTH, 1, 1); cfg.dynamicSmemBytes = smem; cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, direct_tile_kernel<T, NTH, TC, PXT, CH, BOX>, L, (const T*)x, (const T*)w_base, (const T*)w_cond,
                                           bn, delta, (const T*)residual, (T*)y, mask, (float*)p_out, base_only, counters,
                                           div_base, div_cond, div_kw, taps, (uint64_t)0x8000000080000000ull);
  return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}

// Large layers: the layer's channels (at most 64) per block, four channels and two or four pixels per thread.  Small
// ones wait for the chain of additions of one output: one output per thread, 16 channels x 16 pixels per block, so
// that a product costs few instructions and the blocks spread over the SMs.  Measured, us of the bf16 partial sums /
// the fp32 layer with every gate open, for one output, two and four pixels per thread: 100 thousand outputs (4 x 7x7 x
// 512) 44 78 115 / 170 278 395; 201 thousand (56x56 x 64) 13.2 14.8 16.2 / 45 57 54; 401 thousand (2 x 56x56 x 64)
// 24.5 17.7 19.2 / 83 66 70; 803 thousand (4 x 56x56 x 64) 44 18.5 22.1 / 161 74 84; a million (16 x 32x32 x 64)
// 56 29 22 / 203 102 84; 1.6 million (8 x 56x56 x 64) 84 35 36 / 308 144 130.
template <typename T>
int launch_tiles(const LayerDims& L, const void* x, const void* w_base, const void* w_cond, const cg_bn_params& bn,
                 const float* delta, const void* residual, void* y, uint32_t* mask, void* p_out, int base_only,
                 unsigned long long* counters, cudaStream_t stream) {
#define CG_TILE(TC, PXT, CH, ...) launch_tile<T, 256, TC, PXT, CH, ##__VA_ARGS__>(L, taps, x, w_base, w_cond, bn, delta, residual, y, mask, p_out, base_only, counters, stream)
  const int tc = L.c_out <= 16 ? 16 : (L.c_out <= 32 ? 32 : 64);
  const long long outputs = L.m * ((L.c_out + tc - 1) / tc * tc);
  const int v = outputs >= 900000 ? 4 : (outputs >= 250000 ? 2 : 1);
  const TapBox taps = tap_box(L);
  // images smaller than the filter's reach (us with all taps and with the box, before them the kernel of one warp per
  // output: fp32, one pixel x 128 23.2, 5.1, 9.2; 2x2 x 64, 7x7 58, 13.5, 41).  Large layers, where a product of this
  // instance costs four times as much: a fifth of the taps and fewer (4000 x one pixel x 64 53, 13; with 3 of 9 taps
  // 64 x 1x1000 x 32 71, 92)
  if (taps.kh * taps.kw < L.kh * L.kw && (v == 1 || 5 * taps.kh * taps.kw <= L.kh * L.kw)) return CG_TILE(16, 1, 1, true);
  if (v == 1) return CG_TILE(16, 1, 1);
  if (tc == 16) return CG_TILE(16, 2, 4);
  if (tc == 32) return v == 4 ? CG_TILE(32, 4, 4) : CG_TILE(32, 2, 4);
  return v == 4 ? CG_TILE(64, 4, 4) : CG_TILE(64, 2, 4);
#undef CG_TILE
}

}  // namespace

int launch_direct(const LayerDims& L, int in_dtype, const void* x, const void* w_base,
                  const void* w_cond, const cg_bn_params& bn, const float* delta,
                  const void* residual, void* y, uint32_t* mask, void* p_out, int base_only,
                  unsigned long long* counters, cudaStream_t stream) {
  const long long items = L.m * L.words;
  if (items == 0) return 0;
  const int warps_per_block = kThreads / 32;
  long long blocks = (items + warps_per_block - 1) / warps_per_block;
  const long long cap = 148ll * 8 * 8;
  if (blocks > cap) blocks = cap;
  const size_t smem = (size_t)6 * L.c_out * sizeof(float);
  // whole groups of four channels on both paths, and a grid that can be launched
  const bool tiles = L.c_p % 4 == 0 && L.c_r % 4 == 0 && !(L.grouping && L.groups > 1) && L.c_out <= 64 * 65535 &&
                     L.m < (1ll << 31) && (long long)L.ho * L.wo < (1ll << 31) &&
                     (long long)L.kh * L.kw * L.c_in < (1ll << 30);
  if (tiles && in_dtype == CG_F32)
    return launch_tiles<float>(L, x, w_base, w_cond, bn, delta, residual, y, mask, p_out, base_only, counters, stream);
  if (tiles && in_dtype == CG_BF16)
    return launch_tiles<__nv_bfloat16>(L, x, w_base, w_cond, bn, delta, residual, y, mask, p_out, base_only, counters, stream);
  if (in_dtype == CG_F32) {
    direct_gated_conv_kernel<float, float><<<(unsigned)blocks, kThreads, smem, stream>>>(
        L, (const float*)x, (const float*)w_base, (const float*)w_cond, bn, delta,
        (const float*)residual, (float*)y, mask, (float*)p_out, base_only, counters);
  } else if (in_dtype == CG_BF16) {
    direct_gated_conv_kernel<__nv_bfloat16, __nv_bfloat16><<<(unsigned)blocks, kThreads, smem, stream>>>(
        L, (const __nv_bfloat16*)x, (const __nv_bfloat16*)w_base, (const __nv_bfloat16*)w_cond, bn,
        delta, (const __nv_bfloat16*)residual, (__nv_bfloat16*)y, mask, (float*)p_out, base_only,
        counters);
  } else {
    direct_gated_conv_i8_kernel<<<(unsigned)blocks, kThreads, 0, stream>>>(
        L, (const int8_t*)x, (const int8_t*)w_base, (const int8_t*)w_cond, bn, (int8_t*)y, mask,
        (int*)p_out, base_only, counters);
  }
  return (int)cudaGetLastError();
}

// workspace of the channel-wise gate: [partial sums: M x c_out fp32][counts: n x c_out int32]
size_t channel_gate_workspace_bytes(const LayerDims& L) {
  const size_t p_bytes = ((size_t)L.m * L.c_out * sizeof(float) + 255) / 256 * 256;
  return p_bytes + ((size_t)L.n * L.c_out * sizeof(int) + 255) / 256 * 256;
}

int launch_direct_channel_gate(const LayerDims& L, int in_dtype, const void* x, const void* w_base,
                               const void* w_cond, const cg_bn_params& bn, const float* delta,
                               const void* residual, void* y, uint32_t* mask, void* workspace,
                               unsigned long long* counters, cudaStream_t stream) {
  const long long items = L.m * L.words;
  if (items == 0) return 0;
  if (in_dtype != CG_F32 && in_dtype != CG_BF16) return (int)cudaErrorInvalidValue;
  const size_t p_bytes = ((size_t)L.m * L.c_out * sizeof(float) + 255) / 256 * 256;
  float* p_ws = (float*)workspace;
  int* cnt_ws = (int*)((char*)workspace + p_bytes);
  cudaError_t e = cudaMemsetAsync(cnt_ws, 0, (size_t)L.n * L.c_out * sizeof(int), stream);
  if (e != cudaSuccess) return (int)e;
  const int warps_per_block = kThreads / 32;
  long long blocks = (items + warps_per_block - 1) / warps_per_block;
  const long long cap = 148ll * 8 * 8;
  if (blocks > cap) blocks = cap;
  const size_t smem = (size_t)6 * L.c_out * sizeof(float);
  // Eq. 4's threshold on the count, in fp32 like the comparison itself
  const float need = L.channel_tau * (float)(L.ho * L.wo);
  for (int pass = 1; pass <= 2; ++pass) {
    if (in_dtype == CG_F32) {
      direct_gated_conv_kernel<float, float><<<(unsigned)blocks, kThreads, smem, stream>>>(
          L, (const float*)x, (const float*)w_base, (const float*)w_cond, bn, delta,
          (const float*)residual, (float*)y, mask, p_ws, 0, counters, pass, cnt_ws, need);
    } else {
      direct_gated_conv_kernel<__nv_bfloat16, __nv_bfloat16><<<(unsigned)blocks, kThreads, smem, stream>>>(
          L, (const __nv_bfloat16*)x, (const __nv_bfloat16*)w_base, (const __nv_bfloat16*)w_cond, bn,
          delta, (const __nv_bfloat16*)residual, (__nv_bfloat16*)y, mask, p_ws, 0, counters, pass,
          cnt_ws, need);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
  }
  return 0;
}

}  // namespace cg
