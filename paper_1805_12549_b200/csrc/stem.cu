// The stem of a ResNet -- 7x7, stride 2, padding 3, 3 -> 64 channels -- as one kernel from the image to the
// activations.  As a patch matrix and a 1x1 layer over it, batch 128 at 224x224 moved 616 MB out and in again:
// 0.43 ms for the matrix and 0.15 ms for the layer.  Here the patches exist in shared memory only.
//
// A job is up to 128 pixels of one output row.  Its seven input rows are staged in shared memory, zero outside the
// image; the 21 values of a pixel's filter row are consecutive there, 6 elements further on per pixel.  Eight warps
// gather them into the MMA's A tile [pixel][K], K = 7 filter rows of 24 (21 and three zeros: three 16-byte pieces)
// and one zero piece: 11 MMAs of 128 x 64 x 16.  The zeros are real zeros on both sides: no other pixel's value,
// finite or not, meets a zero weight.  Bound by instructions: issue slots 68 % busy (loads and their index arithmetic,
// funnel shifts, epilogue), shared memory 37 %, tensor pipe 11 %, DRAM 9 % at batch 64.
//
// Warps (896 threads): 0 = MMA issuer, 4-11 = epilogue (TMEM lane quadrant x 32 channels, constants in
// registers, as in the window kernel), 12-19 and 20-27 = gather of the even and the odd jobs, each group with an A
// tile and two sets of staged rows of its own (one group alone, its chain of loads, staging and gather exposed
// per job: 192 us at batch 128; two: 183); two accumulators.
// Every wait is bounded.
#include <cstring>

#include "ptx.cuh"
#include "stem.cuh"

namespace cg {

namespace {

constexpr int kThreads = 896, kEpiWarp0 = 4, kEpiWarps = 8, kGatherWarp0 = 12, kGatherWarps = 8;   // (two gather groups)
constexpr int kRowWords = 3 * 127 + 11;               // staged 4-byte words of an input row: 128 pixels
constexpr int kRowsWords = 7 * kRowWords;
constexpr int kLoads = (kRowsWords + kGatherWarps * 32 - 1) / (kGatherWarps * 32);
constexpr uint32_t kATile = 3 * 128 * 128, kBTile = (uint32_t)kStemWeightBytes;
constexpr unsigned kOffB = 2048, kOffA = kOffB + kBTile, kOffRows = kOffA + 2 * kATile;
static_assert(kOffA % 1024 == 0 && kOffB % 1024 == 0, "swizzled tiles");
constexpr unsigned kSmem = kOffRows + 4 * kRowsWords * 4 + 1024;
constexpr int kSpinLimit = 1 << 21;
constexpr long long kWaitCycles = 2000000000ll;

struct SharedS {
  uint64_t a_full[2], a_empty[2], acc_full[2], acc_empty[2], b_ready;
  uint32_t tmem_base, abort_flag, active, rows_active;
  float t[64];
  float4 k[64];                                       // {a1, b1, a2, b2}
};
static_assert(sizeof(SharedS) <= kOffB, "barrier block");

__device__ __noinline__ bool wait_slow(SharedS* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  const long long t0 = clock64();
  for (int i = 0; i < kSpinLimit; ++i) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    if ((i & 15) == 15) {
      if (*(volatile uint32_t*)&sh->abort_flag) return false;
      if (clock64() - t0 > kWaitCycles) break;
    }
  }
  if (atomicCAS(&counters[CNT_STATUS], 0ull, (unsigned long long)CG_ERR_DEVICE_TIMEOUT) == 0ull)
    atomicExch(&counters[CNT_SITE], (unsigned long long)(500 + site));
  atomicExch(&sh->abort_flag, 1u);
  return false;
}

__device__ __forceinline__ bool wait_one(SharedS* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  return ptx::mbar_try_wait(bar, parity, 0u) || wait_slow(sh, counters, bar, parity, site);
}
__device__ __forceinline__ bool wait_warp(SharedS* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  bool ok = ptx::mbar_try_wait(bar, parity, 0u);
  if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, wait_slow(sh, counters, bar, parity, site));
  return ok;
}

// The filter as three K-major tiles [64 rows][128 bytes] in the 128-byte swizzle; rows in the channel order that
// gives an accumulator fragment eight consecutive channels (row 8k + 2q + e of 32 = channel 8q + 2k + e).
__global__ void stem_weights_kernel(const __nv_bfloat16* __restrict__ w, int k_pad, uint4* __restrict__ out) {
  ptx::grid_launch_dependents();
  ptx::grid_dependency_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;   // piece: tile, row, 16-byte piece of the row
  if (i >= 3 * 64 * 8) return;
  const int q = i / 512, row = (i / 8) % 64, pp = i % 8, p = q * 8 + pp, r = p / 3, j = (p % 3) * 8;
  const int ch = (row & ~31) + 8 * ((row >> 1) & 3) + 2 * ((row >> 3) & 3) + (row & 1);
  __align__(16) __nv_bfloat16 v[8];
#pragma unroll
  for (int e = 0; e < 8; ++e)
    v[e] = r < 7 && j + e < 21 ? w[(size_t)ch * k_pad + r * 21 + j + e] : __float2bfloat16(0.f);
  out[q * 512 + row * 8 + (pp ^ (row & 7))] = *reinterpret_cast<const uint4*>(v);
}

struct StemParams {
  const unsigned short* x;
  const uint4* weights;
  __nv_bfloat16* y;
  cg_bn_params bn;
  const float* delta;
  unsigned long long* counters;
  float eps;
  int relu, h, w, ho, wo, segs, jobs;                 // segs: jobs per output row
};

// EVEN: an even image width, whose rows start on 4-byte boundaries
template <bool EVEN>
__global__ void __launch_bounds__(kThreads, 1) stem_kernel(const __grid_constant__ StemParams P) {
  extern __shared__ uint8_t smem_raw[];
  ptx::grid_launch_dependents();
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  SharedS* sh = (SharedS*)smem;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int jobs = (P.jobs - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;   // (grid <= jobs)
  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sh->a_full[i], kGatherWarps); ptx::mbar_init(&sh->a_empty[i], 1);
      ptx::mbar_init(&sh->acc_full[i], 1); ptx::mbar_init(&sh->acc_empty[i], kEpiWarps);
    }
    ptx::mbar_init(&sh->b_ready, 2 * kGatherWarps);
    sh->abort_flag = 0; sh->active = 0; sh->rows_active = 0;
    ptx::fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) ptx::tmem_alloc(&sh->tmem_base, 128);
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  ptx::grid_dependency_wait();
  const uint32_t tmem = sh->tmem_base;
  // job j of this CTA: output row `oh` of image `img`, pixels [ow0, ow0 + cnt)
  auto job_at = [&](int j, int& img, int& oh, int& ow0, int& cnt) {
    const int id = (int)blockIdx.x + j * (int)gridDim.x, row = id / P.segs;
    ow0 = (id - row * P.segs) * 128;
    img = row / P.ho; oh = row - img * P.ho;
    cnt = min(128, P.wo - ow0);
  };

  if (warp == 0) {
    // ============================================================ MMA issuer
    if (ptx::elect_one()) {
      const uint32_t idesc = ptx::idesc_bf16(128, 64), hi = (uint32_t)(ptx::smem_desc(0, 1024, 2) >> 32);
      const uint32_t a0 = (ptx::smem_u32(smem + kOffA) >> 4) | 0x10000u, b0 = (ptx::smem_u32(smem + kOffB) >> 4) | 0x10000u;
      bool ok = wait_one(sh, P.counters, &sh->b_ready, 0, 1);
      for (int j = 0; j < jobs && ok; ++j) {
        const int s = j & 1;
        const uint32_t par = (uint32_t)(j >> 1) & 1u;
        ok = wait_one(sh, P.counters, &sh->acc_empty[s], par ^ 1u, 2) && wait_one(sh, P.counters, &sh->a_full[s], par, 3);
        if (!ok) break;
        ptx::tc_fence_after();
#pragma unroll
        for (int k = 0; k < 11; ++k)
          ptx::umma_bf16(tmem + (uint32_t)s * 64u, ((uint64_t)hi << 32) | (a0 + (uint32_t)s * (kATile >> 4) + (k / 4) * 1024u + (k % 4) * 2u),
                         ((uint64_t)hi << 32) | (b0 + (k / 4) * 512u + (k % 4) * 2u), idesc, k ? 1u : 0u);
        ptx::umma_commit(&sh->a_empty[s]);
        ptx::umma_commit(&sh->acc_full[s]);
      }
    }
    __syncwarp();
  } else if (warp >= kGatherWarp0) {
    // ============================================================ gather
    const int group = (warp - kGatherWarp0) / kGatherWarps, gt = ((int)threadIdx.x - kGatherWarp0 * 32) % (kGatherWarps * 32);
    uint4* s_b = (uint4*)(smem + kOffB);
#pragma unroll
    for (int i = 0; i < (int)(kBTile / 16) / (2 * kGatherWarps * 32); ++i) {
      const int id = gt + (2 * i + group) * kGatherWarps * 32;
      s_b[id] = P.weights[id];
    }
    ptx::fence_proxy_async();
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive(&sh->b_ready);
    uint32_t v[kLoads];
    // words of the job's input rows: word q of row r holds the row's elements 6*ow0 - 10 + 2q and the next.  All
    // loads of a job are issued before any result is used (out-of-range ones read the first word of x).
    uint32_t valid = 0;
    auto fetch = [&](int j) {
      int img, oh, ow0, cnt;
      job_at(j, img, oh, ow0, cnt);
      const int words = 3 * (cnt - 1) + 11, w3 = P.w * 3;
      valid = 0;
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        const int id = gt + i * kGatherWarps * 32, r = id / kRowWords, q = id - r * kRowWords;
        const int yy = 2 * oh + r - 3, e = 6 * ow0 + 2 * q - 10;
        const bool in = r < 7 && q < words && yy >= 0 && yy < P.h && e >= 0 && e < w3;
        const unsigned short* p = P.x + (in ? ((long long)img * P.h + yy) * w3 + e : 0);
        if (EVEN) {
          v[i] = *(const uint32_t*)p;           // (rows of an even number of elements: whole words)
        } else {
          const uint32_t a = *p, b = in && e + 1 < w3 ? p[1] : 0;
          v[i] = a | b << 16;
        }
        valid |= in ? 1u << i : 0u;
      }
    };
    const int px = gt & 127, upper = gt >> 7;         // a thread gathers filter rows 0-3 or 4-6 of a pixel
    bool ok = true;
    if (group < jobs) fetch(group);
    for (int j = group; j < jobs && ok; j += 2) {
      const int s = j & 1;
      uint32_t* rows = (uint32_t*)(smem + kOffRows) + (group * 2 + ((j >> 1) & 1)) * kRowsWords;   // (warps may still gather the other)
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        const int id = gt + i * kGatherWarps * 32;
        if (id < kRowsWords) rows[id] = (valid >> i) & 1u ? v[i] : 0u;
      }
      ok = wait_warp(sh, P.counters, &sh->a_empty[s], ((uint32_t)(j >> 1) & 1u) ^ 1u, 4);
      // the staged rows are complete; a warp whose wait gave up takes its siblings with it
      if (ptx::named_bar_or(3 + group, kGatherWarps * 32, !ok)) break;
      if (j + 2 < jobs) fetch(j + 2);                 // (in flight during the gather)
      uint8_t* a = smem + kOffA + s * kATile + px * 128;
      auto put = [&](int piece, const uint4& d) {
        *(uint4*)(a + (piece >> 3) * (128 * 128) + (((piece & 7) ^ (px & 7)) << 4)) = d;
      };
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = upper * 4 + i;
        if (r >= 7) { put(21, make_uint4(0u, 0u, 0u, 0u)); break; }
        // 21 elements from the upper half of the pixel's first word on
        const uint32_t* src = rows + r * kRowWords + 3 * px;
        uint32_t m[11], o[11];
#pragma unroll
        for (int k = 0; k < 11; ++k) m[k] = src[k];
#pragma unroll
        for (int k = 0; k < 10; ++k) o[k] = __funnelshift_r(m[k], m[k + 1], 16);
        o[10] = m[10] >> 16;
        put(3 * r, make_uint4(o[0], o[1], o[2], o[3]));
        put(3 * r + 1, make_uint4(o[4], o[5], o[6], o[7]));
        put(3 * r + 2, make_uint4(o[8], o[9], o[10], 0u));
      }
      ptx::fence_proxy_async();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&sh->a_full[s]);
    }
  } else if (warp >= kEpiWarp0) {
    // ============================================================ epilogue
    const int et = (int)threadIdx.x - kEpiWarp0 * 32;
    if (et < 64) {
      const ChannelConsts k = fold_channel(P.bn, P.delta, P.eps, et);
      sh->t[et] = k.t; sh->k[et] = make_float4(k.a1, k.b1, k.a2, k.b2);
    }
    ptx::named_bar_sync(2, kEpiWarps * 32);
    const int quad = warp & 3, c0 = ((warp - kEpiWarp0) >> 2) * 32, q8 = (lane & 3) * 8, r4 = lane >> 2;
    float t[8];
    float4 k[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) { t[e] = sh->t[c0 + q8 + e]; k[e] = sh->k[c0 + q8 + e]; }
    uint32_t active = 0, rows_active = 0;               // (rows: of all four lanes of a row, kept by every lane)
    bool ok = true;
    for (int j = 0; j < jobs && ok; ++j) {
      const int s = j & 1;
      int img, oh, ow0, cnt;
      job_at(j, img, oh, ow0, cnt);
      __nv_bfloat16* yp = P.y + (((long long)img * P.ho + oh) * P.wo + ow0) * 64 + c0 + q8;
      ok = wait_warp(sh, P.counters, &sh->acc_full[s], (uint32_t)(j >> 1) & 1u, 5);
      if (!ok) break;
      ptx::tc_fence_after();
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        uint32_t p[2][8];
        const uint32_t tp = tmem + ((uint32_t)(quad * 32 + 16 * i) << 16) + (uint32_t)(s * 64 + c0);
        __syncwarp();                                 // (the loads are .aligned; the rows of a ragged tile diverge)
        ptx::tmem_ld_frag16(tp, p[0]);
        ptx::tmem_ld_frag16(tp + 16, p[1]);
        ptx::tmem_ld_wait16(p[0], p[1]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row = quad * 32 + 16 * i + 8 * h + r4;
          uint32_t out[4], fired = 0;
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            float v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int c = 2 * g + e;
              const float pv = __uint_as_float(p[g >> 1][4 * (g & 1) + 2 * h + e]);
              const bool d = pv >= t[c];              // (a NaN sum does not fire)
              fired += d ? 1u : 0u;
              v[e] = fmaf(d ? k[c].z : k[c].x, pv, d ? k[c].w : k[c].y);
            }
            if (P.relu) { v[0] = fmaxf(v[0], 0.f); v[1] = fmaxf(v[1], 0.f); }
            const __nv_bfloat162 b = __floats2bfloat162_rn(v[0], v[1]);
            out[g] = *reinterpret_cast<const uint32_t*>(&b);
          }
          if (row < cnt) *(uint4*)(yp + (long long)row * 64) = make_uint4(out[0], out[1], out[2], out[3]);
          else fired = 0;
          active += fired;
          uint32_t on = __ballot_sync(0xffffffffu, fired != 0u);   // four lanes to a row
          on |= on >> 1; on |= on >> 2;
          rows_active += (uint32_t)__popc(on & 0x11111111u);
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&sh->acc_empty[s]);
    }
    active = __reduce_add_sync(0xffffffffu, active);
    if (lane == 0) { atomicAdd(&sh->active, active); atomicAdd(&sh->rows_active, rows_active); }
  }
  __syncwarp();
  if (*(volatile uint32_t*)&sh->abort_flag) {
    const long long t_drain = clock64();              // let MMAs in flight finish
    while (clock64() - t_drain < 4000000ll) {}
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  if (threadIdx.x == 0 && !*(volatile uint32_t*)&sh->abort_flag) {
    if (sh->active) atomicAdd(&P.counters[CNT_ACTIVE], (unsigned long long)sh->active);
    if (sh->rows_active) atomicAdd(&P.counters[CNT_ROWS_ACTIVE], (unsigned long long)sh->rows_active);
    if (blockIdx.x == 0) {
      atomicAdd(&P.counters[CNT_CALLS], 1ull);
      atomicAdd(&P.counters[CNT_ROWS_TOTAL], (unsigned long long)(P.jobs / P.segs) * P.wo * 2ull);
      atomicAdd(&P.counters[CNT_EXEC_MACS], (unsigned long long)P.jobs * 128ull * 64ull * 176ull);
    }
  }
  if (warp == 0) {
    __syncwarp();
    ptx::tmem_dealloc(tmem, 128);
  }
}

}  // namespace

int launch_stem(const void* x, int n, int h, int w, const void* w_base, int k_pad, const cg_bn_params& bn,
                const float* delta, float eps, int relu, void* y, void* ws, unsigned long long* counters,
                cudaStream_t stream) {
  StemParams P;
  P.x = static_cast<const unsigned short*>(x); P.weights = static_cast<const uint4*>(ws);
  P.y = static_cast<__nv_bfloat16*>(y); P.bn = bn; P.delta = delta; P.counters = counters; P.eps = eps; P.relu = relu;
  P.h = h; P.w = w; P.ho = (h - 1) / 2 + 1; P.wo = (w - 1) / 2 + 1;
  P.segs = (P.wo + 127) / 128;
  const long long jobs = (long long)n * P.ho * P.segs;
  if (jobs > 0x3fffffffll) return (int)cudaErrorInvalidValue;
  P.jobs = (int)jobs;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 148;
  static bool set[64][2] = {};
  void (*kernel)(StemParams) = w % 2 == 0 ? stem_kernel<true> : stem_kernel<false>;
  if (!set[dev][w % 2]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return (int)e;
    set[dev][w % 2] = true;
  }
  static_assert(kSmem <= 227 * 1024, "shared memory");
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3(12, 1, 1);
  cfg.blockDim = dim3(128, 1, 1);
  cudaError_t e = cudaLaunchKernelEx(&cfg, stem_weights_kernel, static_cast<const __nv_bfloat16*>(w_base), k_pad, static_cast<uint4*>(ws));
  if (e != cudaSuccess) return (int)e;
  cfg.gridDim = dim3((unsigned)(jobs < sms ? jobs : sms), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = 227 * 1024;                  // (as the layer kernels: no reconfiguration between them)
  e = cudaLaunchKernelEx(&cfg, kernel, P);
  return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}

}  // namespace cg
