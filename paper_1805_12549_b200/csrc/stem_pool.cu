// The stem of a ResNet and the max pooling behind it -- 7x7, stride 2, padding 3, 3 -> 64 channels, then 3x3, stride 2,
// padding 1 -- as one kernel from the image to both activations, for batches that fill the SMs.
//
// The separate stem kernel (stem.cu) gathers every pixel's 7x7x3 patch into an MMA operand: 34 instructions per output,
// 183 us at batch 128 of 224x224, and the pooling reads the 205 MB again (45 us).  Here nothing is gathered.  With its
// pixels padded to four channels (8 bytes), an image row is an operand already: output pixel ow needs the pixels
// 2*ow - 3 .. 2*ow + 3 of a row, four 16-byte pieces of two pixels, and the next output pixel's start one piece further on.
// In the unswizzled K-major layout (8 rows x 16 bytes, consecutive) row m of an MMA's A operand may lie 16 bytes behind row
// m - 1, so that neighbouring rows share their pieces: A is the staged row read with two pieces to a K step, 14 steps for
// the 7 filter rows.  Piece i holds the pixels 2i - 3 and 2i - 2; the last piece of a window, whose second pixel belongs to
// no tap, comes from a copy in which that pixel is zero: no pixel's value, finite or not, meets a zero weight.
//
// Pooled column e needs the output columns 2e - 1, 2e and 2e + 1.  Even and odd columns are separate MMAs (pieces of even
// and odd number are separate arrays), so accumulator row l holds column 2e in the one and 2e + 1 in the other, and the
// neighbour 2e - 1 is the odd column of row l - 1.  The 8-row groups of an operand are 160 bytes apart, each with its own ten
// pieces: a group's first row repeats the last one of the group before, and the other seven find their neighbour in
// the same group, one shuffle away.  16 groups: two strips of 8 x 7 = 56 pooled columns, each strip walking down its image.
//
// A unit of work is one pooled row of both strips: the output rows a = 2ph and b = 2ph + 1 from nine input rows.  An input
// row serves a with filter row k and b with k - 2, and the filter is stored so that both are one B operand of N = 128.
// Vertically the maximum runs in registers; the row 2ph - 1 is the last unit's b (a strip starts with a unit for that row).
//
// Warps (640 threads): 0 = MMA issuer, 4-19 = epilogue (16 TMEM lanes x 32 channels each: batch norm, activation, both
// stores), 1-3 = staging, four input rows of both strips per unit into a ring of 16 rows; a thread's pieces are the same
// ones in every row, so that a unit has no index arithmetic (with it, in four warps, batch 128 took 114 us).
// Every wait is bounded.
//
// A unit takes 6,000 cycles, 2,100 of MMAs: the epilogue bounds it, half of it (the units without stores take 1,500 for half
// the rows) by getting its stores out; 128 images of 224x224 move 295 MB (45 us at the copy rate) in 98 us.
#include <cstring>

#include "ptx.cuh"
#include "stem.cuh"

namespace cg {

namespace {

constexpr int kThreads = 640, kEpiWarp0 = 4, kEpiWarps = 16, kStageWarps = 3;   // (with more the epilogue's registers do not fit)
constexpr int kStageThreads = kStageWarps * 32, kPieces = 16 * 10;                 // (strip, group, piece) of a row
constexpr uint32_t kGroup = 160, kArray = 16 * kGroup, kRow = 4 * kArray;          // bytes; arrays: even, odd, their copies
constexpr uint32_t kPe = 0, kPo = kArray, kQe = 2 * kArray, kQo = 3 * kArray;      // (Q: second pixel zero)
constexpr uint32_t kPiece = 7 * 1024;                                              // filter: one piece of all filter rows
constexpr unsigned kOffB = 2048, kOffA = kOffB + 5 * kPiece, kSmem = kOffA + 16 * kRow + 1024;
static_assert(kSmem <= 227 * 1024 && 2 * kStageThreads >= kPieces, "shared memory");
constexpr int kCols = 56;                              // pooled columns of a strip
constexpr int kSpinLimit = 1 << 21;
constexpr long long kWaitCycles = 2000000000ll;

struct SharedP {
  uint64_t full[4], empty[4], acc_full[2], acc_empty[2];
  uint32_t tmem_base, abort_flag, active, rows_active;
  float t[64];
  float4 k[64];                                        // {a1, b1, a2, b2}
};
static_assert(sizeof(SharedP) <= kOffB, "barrier block");

struct StemPoolParams {
  const uint32_t* x;
  const __nv_bfloat16* w;
  __nv_bfloat16 *y, *pooled;
  cg_bn_params bn;
  const float* delta;
  unsigned long long* counters;
  float eps;
  int relu, k_pad, h, w2, ho, wo, hp, wp;              // w2: 4-byte words of an image row
  int strips, col_tiles, segs, per;                    // strip = (image * col_tiles + column tile) * segs + segment of `per` rows
  int items;                                           // pairs of strips
};

__device__ __noinline__ bool wait_slow(SharedP* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  const long long t0 = clock64();
  for (int i = 0; i < kSpinLimit; ++i) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    if ((i & 15) == 15) {
      if (*(volatile uint32_t*)&sh->abort_flag) return false;
      if (clock64() - t0 > kWaitCycles) break;
    }
  }
  if (atomicCAS(&counters[CNT_STATUS], 0ull, (unsigned long long)CG_ERR_DEVICE_TIMEOUT) == 0ull)
    atomicExch(&counters[CNT_SITE], (unsigned long long)(600 + site));
  atomicExch(&sh->abort_flag, 1u);
  return false;
}
__device__ __forceinline__ bool wait_one(SharedP* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  return ptx::mbar_try_wait(bar, parity, 0u) || wait_slow(sh, counters, bar, parity, site);
}
__device__ __forceinline__ bool wait_warp(SharedP* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity, int site) {
  bool ok = ptx::mbar_try_wait(bar, parity, 0u);
  if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, wait_slow(sh, counters, bar, parity, site));
  return ok;
}

// Low word of an unswizzled K-major operand descriptor: start, and the distance `lbo` of a K step's two pieces.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) { return (addr >> 4) | (lbo >> 4) << 16; }
// Its high word: 8-row groups `sbo` apart.
constexpr uint32_t desc_hi(uint32_t sbo) { return (sbo >> 4) | 1u << 14; }

// Where filter row r lies within a piece: rows of one parity together, descending, so that the 64 channels of row r are
// followed by those of r - 2.
__host__ __device__ constexpr uint32_t filter_at(int r) { return (uint32_t)(r % 2 == 0 ? (6 - r) / 2 : 4 + (5 - r) / 2) * 1024u; }

__device__ __forceinline__ uint32_t max2(uint32_t a, uint32_t b) {
  const __nv_bfloat162 r = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
  return *reinterpret_cast<const uint32_t*>(&r);
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// The same of max(v, 0), for numbers (of a NaN it makes a NaN).
__device__ __forceinline__ uint32_t pack2_relu(float a, float b) {
  uint32_t v;
  asm("cvt.rn.relu.bf16x2.f32 %0, %1, %2;" : "=r"(v) : "f"(b), "f"(a));
  return v;
}

__global__ void __launch_bounds__(kThreads, 1) stem_pool_kernel(const __grid_constant__ StemPoolParams P) {
  extern __shared__ uint8_t smem_raw[];
  ptx::grid_launch_dependents();
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  SharedP* sh = (SharedP*)smem;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int units = P.per + 1;
  if (threadIdx.x == 0) {
    for (int i = 0; i < 4; ++i) { ptx::mbar_init(&sh->full[i], kStageWarps); ptx::mbar_init(&sh->empty[i], 1); }
    for (int i = 0; i < 2; ++i) { ptx::mbar_init(&sh->acc_full[i], 1); ptx::mbar_init(&sh->acc_empty[i], kEpiWarps); }
    sh->abort_flag = 0; sh->active = 0; sh->rows_active = 0;
    ptx::fence_mbar_init();
  }
  __syncwarp();
  if (warp == 0) ptx::tmem_alloc(&sh->tmem_base, 512);
  ptx::grid_dependency_wait();
  // The filter, by way of the ring's room: read element by element where it is put together, the set-up took 15,000 cycles.
  uint4* s_w = (uint4*)(smem + kOffA);                 // [64][152] elements of the 147
  for (int i = threadIdx.x; i < 64 * 19; i += kThreads) s_w[i] = *((const uint4*)(P.w + (size_t)(i / 19) * P.k_pad) + i % 19);
  __syncthreads();
  // Piece p of row r and channel ch is the taps 2p and 2p + 1 with four channels each, the fourth (and tap 7) zero.  Pieces in
  // the order 0, 1, 0, 2, 3 (the odd columns' first step takes 1 before 0); channels of a block of 32 in the order that gives
  // an accumulator fragment eight consecutive ones (row 8k + 2q + e = channel 8q + 2k + e).
  for (int i = (int)threadIdx.x; i < 5 * 7 * 64; i += kThreads) {
    const int row = i & 63, r = (i >> 6) % 7, slot = (i >> 6) / 7, p = slot < 2 ? slot : slot == 2 ? 0 : slot - 1;
    const int ch = (row & ~31) + 8 * ((row >> 1) & 3) + 2 * ((row >> 3) & 3) + (row & 1);
    const __nv_bfloat16* src = (const __nv_bfloat16*)s_w + ch * 152 + r * 21 + p * 6;
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = (e & 3) < 3 && (p < 3 || e < 4) ? src[(e >> 2) * 3 + (e & 3)] : __float2bfloat16(0.f);
    *(uint4*)(smem + kOffB + slot * kPiece + filter_at(r) + row * 16) = *reinterpret_cast<const uint4*>(v);
  }
  if (threadIdx.x >= kThreads - 64) {
    const int c = (int)threadIdx.x - (kThreads - 64);
    const ChannelConsts k = fold_channel(P.bn, P.delta, P.eps, c);
    sh->t[c] = k.t; sh->k[c] = make_float4(k.a1, k.b1, k.a2, k.b2);
  }
  ptx::fence_proxy_async();
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sh->tmem_base;
  // strip s of an item: image, first pooled row, first pooled column
  auto strip_at = [&](int item, int s, int& img, int& p0, int& col0) {
    const int id = item * 2 + s, row = id / P.segs;
    img = row / P.col_tiles;
    p0 = (id - row * P.segs) * P.per;
    col0 = (row - img * P.col_tiles) * kCols;
    return id < P.strips;
  };

  if (warp == 0) {
    // ============================================================ MMA issuer
    if (ptx::elect_one()) {
      const uint32_t a_ring = ptx::smem_u32(smem + kOffA), b0 = ptx::smem_u32(smem + kOffB);
      constexpr uint64_t a_hi = (uint64_t)desc_hi(kGroup) << 32, b_hi = (uint64_t)desc_hi(128) << 32;
      constexpr uint32_t id64 = ptx::idesc_bf16(128, 64), id128 = ptx::idesc_bf16(128, 128);
      unsigned g = 0, n = 0;                           // row groups and units so far
      bool ok = true;
      for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
        for (int u = 0; u < units; ++u, ++g, ++n) {
          if (u == 0)
            ok = wait_one(sh, P.counters, &sh->full[g & 3], (g >> 2) & 1, 1) &&
                 wait_one(sh, P.counters, &sh->full[(g + 1) & 3], ((g + 1) >> 2) & 1, 1);
          ok = ok && wait_one(sh, P.counters, &sh->full[(g + 2) & 3], ((g + 2) >> 2) & 1, 1) &&
               wait_one(sh, P.counters, &sh->acc_empty[n & 1], ((n >> 1) & 1) ^ 1, 2);
          if (!ok) break;
          ptx::tc_fence_after();
#pragma unroll 1
          for (int odd = 0; odd < 2; ++odd) {
            const uint32_t d = tmem + (n & 1) * 256u + (uint32_t)odd * 128u;
            // the two K steps of a filter row: pieces (0, 1) and (2, 3) of the even columns, (1, 0) and (2, 3) of the odd ones
            const uint32_t a1 = odd ? desc_lo(kPe + 16, kPo - kPe - 16) : desc_lo(kPe, kPo - kPe);
            const uint32_t a2 = odd ? desc_lo(kPo + 16, kQe - kPo + 16) : desc_lo(kPe + 16, kQo - kPe);
            const uint32_t b1 = desc_lo(b0 + (odd ? kPiece : 0u), kPiece), b2 = desc_lo(b0 + 3 * kPiece, kPiece);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              const int k = i < 5 ? i + 2 : i < 7 ? i - 5 : i;   // input rows 2-6 (both output rows), 0, 1 (a), 7, 8 (b)
              const uint32_t row = (a_ring + (((g + (unsigned)(k / 4)) & 3) * 4u + (unsigned)(k % 4)) * kRow) >> 4;
              const uint32_t dk = d + (k > 6 ? 64u : 0u), f = filter_at(k > 6 ? k - 2 : k) >> 4, idesc = i < 5 ? id128 : id64;
              ptx::umma_bf16(dk, a_hi | (a1 + row), b_hi | (b1 + f), idesc, i ? 1u : 0u);
              ptx::umma_bf16(dk, a_hi | (a2 + row), b_hi | (b2 + f), idesc, 1u);
            }
          }
          ptx::umma_commit(&sh->empty[g & 3]);
          ptx::umma_commit(&sh->acc_full[n & 1]);
        }
        if (!ok) break;
        ptx::umma_commit(&sh->empty[g & 3]);
        ptx::umma_commit(&sh->empty[(g + 1) & 3]);
        g += 2;
      }
    }
    __syncwarp();
  } else if (warp < kEpiWarp0) {
    // ============================================================ staging
    // Piece t of group gr of a strip: the pixels 4e - 3 .. 4e of column e = 7 * gr - 1 + t, words 6e - 5 .. 6e + 1 of the row.
    // A thread has one piece or two.
    const int st = (int)threadIdx.x - 32;
    uint32_t v[2][4][7];                               // the words of four rows
    uint32_t inside[2] = {0, 0};                       // which of a row's lie in the image
    const uint32_t* src[2] = {nullptr, nullptr};
    int y0[2] = {0, 0};                                // first row of the item's first group
    auto start = [&](int item) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int q = st + i * kStageThreads, s = q / 80, e80 = q - s * 80;
        int img, p0, col0;
        const bool in = q < kPieces && strip_at(item, s, img, p0, col0);
        inside[i] = 0;
        if (!in) continue;
        const int k0 = 6 * (col0 + 7 * (e80 / 10) - 1 + e80 % 10) - 5;
        y0[i] = 4 * (p0 - 1) - 3;
        src[i] = P.x + (long long)img * P.h * P.w2 + k0;
#pragma unroll
        for (int j = 0; j < 7; ++j) inside[i] |= (unsigned)(k0 + j) < (unsigned)P.w2 ? 1u << j : 0u;
      }
    };
    auto fetch = [&](int gi) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int yy = y0[i] + 4 * gi + r;
          const uint32_t* row = src[i] + (long long)yy * P.w2;
          const uint32_t on = yy >= 0 && yy < P.h ? inside[i] : 0u;
#pragma unroll
          for (int j = 0; j < 7; ++j) {
            v[i][r][j] = 0;
            if ((on >> j) & 1u) v[i][r][j] = row[j];
          }
        }
    };
    unsigned g = 0;
    bool ok = true;
    if ((int)blockIdx.x < P.items) { start(blockIdx.x); fetch(0); }
    for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
      for (int gi = 0; gi < units + 2; ++gi, ++g) {
        ok = wait_warp(sh, P.counters, &sh->empty[g & 3], ((g >> 2) & 1) ^ 1, 3);
        if (!ok) break;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int q = st + i * kStageThreads;
          if (q >= kPieces) break;
          uint8_t* dst = smem + kOffA + (g & 3) * 4u * kRow + (q / 10) * kGroup + (q % 10) * 16;
#pragma unroll
          for (int r = 0; r < 4; ++r, dst += kRow) {
            uint32_t w[6];                             // twelve elements from the upper half of the first word on
#pragma unroll
            for (int j = 0; j < 6; ++j) w[j] = __funnelshift_r(v[i][r][j], v[i][r][j + 1], 16);
            // pixels {0 1 2} {3 4 5} {6 7 8} {9 10 11} to four channels each
            const uint32_t p0b = w[1] & 0xffffu, p1a = __funnelshift_r(w[1], w[2], 16), p1b = w[2] >> 16;
            const uint32_t p2b = w[4] & 0xffffu, p3a = __funnelshift_r(w[4], w[5], 16), p3b = w[5] >> 16;
            *(uint4*)(dst + kPe) = make_uint4(w[0], p0b, p1a, p1b);
            *(uint4*)(dst + kPo) = make_uint4(w[3], p2b, p3a, p3b);
            *(uint4*)(dst + kQe) = make_uint4(w[0], p0b, 0u, 0u);
            *(uint4*)(dst + kQo) = make_uint4(w[3], p2b, 0u, 0u);
          }
        }
        ptx::fence_proxy_async();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh->full[g & 3]);
        // the next rows are on their way while this warp waits for a free slot
        if (gi + 1 < units + 2) fetch(gi + 1);
        else if (item + (int)gridDim.x < P.items) { start(item + gridDim.x); fetch(0); }
      }
    }
  } else {
    // ============================================================ epilogue
    const int quad = warp & 3, sub = (warp - kEpiWarp0) >> 2, half = sub & 1, c0 = (sub >> 1) * 32;
    const int q8 = (lane & 3) * 8, l = lane >> 2;
    const int s = quad >> 1;                           // strip
    const int e_in = 7 * ((quad & 1) * 4 + half * 2) - 1 + l;   // pooled column within the strip (the second row: 7 further)
    uint64_t a1[4], b1[4];                             // pairs of channels
    bool shut = true;                                  // no finite sum fires
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const float4 k0 = sh->k[c0 + q8 + 2 * o], k1 = sh->k[c0 + q8 + 2 * o + 1];
      a1[o] = ptx::pack_f32x2(k0.x, k1.x); b1[o] = ptx::pack_f32x2(k0.y, k1.y);
    }
    // (and the constants are finite: what finite sums make of them is a number, for the packed activation below)
    for (int c = 0; c < 8; ++c) {
      const float4 k = sh->k[c0 + q8 + c];
      shut = shut && !(sh->t[c0 + q8 + c] < __int_as_float(0x7f800000)) && isfinite(k.x) && isfinite(k.y);
    }
    shut = __all_sync(0xffffffffu, shut);
    const uint32_t ninf = 0xff80ff80u;
    uint32_t active = 0, rows_active = 0;
    unsigned n = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < P.items && ok; item += gridDim.x) {
      int img, p0, col0;
      const bool in = strip_at(item, s, img, p0, col0);
      const int p1 = min(p0 + P.per, P.hp);
      const int e0 = col0 + e_in;                      // columns e0 and e0 + 7
      // bit 2 * odd + h: the fragment's row h has an output column, even or odd, inside the image
      uint32_t cols = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (e0 + 7 * (i & 1) >= 0 && 2 * (e0 + 7 * (i & 1)) + (i >> 1) < P.wo) cols |= 1u << i;
      const bool edge = __any_sync(0xffffffffu, cols != 15u);
      uint32_t carry[2][2][4];                         // row b of the last unit: even and odd columns
#pragma unroll
      for (int i = 0; i < 16; ++i) carry[i >> 3][(i >> 2) & 1][i & 3] = ninf;
      for (int u = 0; u < units; ++u, ++n) {
        const int ph = p0 - 1 + u;
        const bool out = in && u > 0 && ph < p1;       // (the first unit only brings the row above)
        ok = wait_warp(sh, P.counters, &sh->acc_full[n & 1], (n >> 1) & 1, 4);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t tp = tmem + ((uint32_t)(quad * 32 + half * 16) << 16) + (n & 1) * 256u + (uint32_t)c0;
        __nv_bfloat16* y0 = P.y + (((long long)img * P.ho + 2 * ph) * P.wo + 2 * e0) * 64 + c0 + q8;
        uint32_t best[2][4];                           // the window's maximum so far
#pragma unroll
        for (int odd = 1; odd >= 0; --odd) {
          uint32_t top[2][4];                          // of this column's three rows
#pragma unroll
          for (int i = 0; i < 8; ++i) top[i >> 2][i & 3] = carry[odd][i >> 2][i & 3];
#pragma unroll 1
          for (int ab = 0; ab < 2; ++ab) {
            const int row = 2 * ph + ab;
            if (!(in && ph < p1 && row >= 0 && row < P.ho) || (u == 0 && ab == 0)) continue;   // (uniform over the warp)
            const uint32_t tq = tp + (uint32_t)(odd * 128 + ab * 64);
            uint32_t p[2][8], act[2][4];
            __syncwarp();
            ptx::tmem_ld_frag16(tq, p[0]);
            ptx::tmem_ld_frag16(tq + 16, p[1]);
            ptx::tmem_ld_wait16(p[0], p[1]);
            uint64_t bad = 0;                          // 0 * sums: not a number once a sum is infinite
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                const uint64_t v = ptx::pack_f32x2(__uint_as_float(p[o >> 1][4 * (o & 1) + 2 * h]),
                                                   __uint_as_float(p[o >> 1][4 * (o & 1) + 2 * h + 1]));
                bad = ptx::fma_f32x2(v, 0ull, bad);
                float f0, f1;
                ptx::unpack_f32x2(ptx::fma_f32x2(a1[o], v, b1[o]), f0, f1);
                act[h][o] = P.relu ? pack2_relu(f0, f1) : pack2(f0, f1);
              }
            float z0, z1;
            ptx::unpack_f32x2(bad, z0, z1);
            if (!shut || __any_sync(0xffffffffu, !(z0 == 0.f && z1 == 0.f))) {
              // gates that can fire (an infinite sum meets an infinite threshold, a tie): every output from its definition
              __syncwarp();
              ptx::tmem_ld_frag16(tq, p[0]);           // (again, rather than kept in registers for this)
              ptx::tmem_ld_frag16(tq + 16, p[1]);
              ptx::tmem_ld_wait16(p[0], p[1]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                uint32_t fired = 0;
#pragma unroll
                for (int o = 0; o < 4; ++o) {
                  float f[2];
#pragma unroll
                  for (int c = 0; c < 2; ++c) {
                    const float pv = __uint_as_float(p[o >> 1][4 * (o & 1) + 2 * h + c]);
                    const int ch = c0 + q8 + 2 * o + c;
                    const float4 k = sh->k[ch];
                    const bool d = pv >= sh->t[ch];
                    fired += d ? 1u : 0u;
                    f[c] = fmaf(d ? k.z : k.x, pv, d ? k.w : k.y);
                  }
                  act[h][o] = pack2(f[0], f[1]);
                  if (P.relu) act[h][o] = max2(act[h][o], 0u);
                }
                if (!out || l == 0 || !((cols >> (2 * odd + h)) & 1u)) fired = 0;
                active += fired;
                uint32_t on = __ballot_sync(0xffffffffu, fired != 0u);   // four lanes to a pixel
                on |= on >> 1; on |= on >> 2;
                rows_active += (uint32_t)__popc(on & 0x11111111u);
              }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (out && l > 0 && ((cols >> (2 * odd + h)) & 1u))
                __stcs((uint4*)(y0 + (long long)ab * P.wo * 64 + (14 * h + odd) * 64), make_uint4(act[h][0], act[h][1], act[h][2], act[h][3]));
              if (edge && !((cols >> (2 * odd + h)) & 1u)) {
#pragma unroll
                for (int o = 0; o < 4; ++o) act[h][o] = ninf;
              }
#pragma unroll
              for (int o = 0; o < 4; ++o) {
                top[h][o] = max2(top[h][o], act[h][o]);
                if (ab) carry[odd][h][o] = act[h][o];
              }
            }
          }
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int o = 0; o < 4; ++o)
              best[h][o] = odd ? max2(top[h][o], __shfl_up_sync(0xffffffffu, top[h][o], 4)) : max2(best[h][o], top[h][o]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if (out && l > 0 && ((cols >> h) & 1u))      // (a window of NaN gives -inf)
            *(uint4*)(P.pooled + (((long long)img * P.hp + ph) * P.wp + e0 + 7 * h) * 64 + c0 + q8) =
                make_uint4(max2(best[h][0], ninf), max2(best[h][1], ninf), max2(best[h][2], ninf), max2(best[h][3], ninf));
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&sh->acc_empty[n & 1]);
      }
    }
    active = __reduce_add_sync(0xffffffffu, active);
    if (lane == 0 && active) { atomicAdd(&sh->active, active); atomicAdd(&sh->rows_active, rows_active); }
  }
  __syncwarp();
  if (*(volatile uint32_t*)&sh->abort_flag) {
    const long long t_drain = clock64();               // let MMAs in flight finish
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
      atomicAdd(&P.counters[CNT_ROWS_TOTAL], (unsigned long long)(P.strips / (P.col_tiles * P.segs)) * P.ho * P.wo * 2ull);
      atomicAdd(&P.counters[CNT_EXEC_MACS], (unsigned long long)P.items * units * (20ull * 128 + 16ull * 64) * 128 * 16);
    }
  }
  if (warp == 0) {
    __syncwarp();
    ptx::tmem_dealloc(tmem, 512);
  }
}

// Strips of an image: as many segments as make the longest CTA shortest (every segment repeats one unit and fills a ring).
// More than 1024 of them, seven to an SM, are not looked at.
void split_strips(long long columns, int hp, StemPoolPlan* plan) {
  double best = 0.0;
  plan->per = 0;
  for (int s = 1; s <= hp && s <= 1024; ++s) {
    const int per = (hp + s - 1) / s, segs = (hp + per - 1) / per;
    const long long items = (columns * segs + 1) / 2;
    const double cost = (double)((items + plan->sms - 1) / plan->sms) * (per + 1.7);
    if (plan->per == 0 || cost < best) { best = cost; plan->per = per; plan->segs = segs; }
  }
}

}  // namespace

// Measured, us of the stem and the pooling kernel / of this one, 224x224: 1 image 9.4 / 13.0, 2 11.6 / 13.1, 4 15.3 / 13.5, 6 17.2
// / 16.4, 8 20.4 / 16.4, 16 32.5 / 22.1, 32 56.5 / 32.1, 128 229 / 97.6; 32 x 448x448 232 / 97; 64 x 300x300 (two column tiles)
// 286 / 128; 128 x 112x112 (half of a strip's columns) 94 / 48; 200 x 64x64 (a third) 81 / 46.  The line lies at four output
// rows per SM, clear of the edge, and at a quarter of the columns.
bool stem_pool_pays(int n, int h, int w) {
  const long long ho = (h - 1) / 2 + 1, wo = (w - 1) / 2 + 1, cols = (wo + 2 * kCols - 1) / (2 * kCols);
  if (w % 2 || (long long)n * cols * ho > 0x0fffffffll) return false;
  return n * ho >= 148 * 4 && 4 * wo >= 2 * kCols * cols;
}

int launch_stem_pool(StemPoolPlan* plan, const void* x, int n, int h, int w, const void* w_base, int k_pad, const cg_bn_params& bn,
                     const float* delta, float eps, int relu, void* y, void* pooled, unsigned long long* counters,
                     cudaStream_t stream) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  StemPoolParams P;
  std::memset(&P, 0, sizeof(P));
  P.x = static_cast<const uint32_t*>(x); P.w = static_cast<const __nv_bfloat16*>(w_base);
  P.y = static_cast<__nv_bfloat16*>(y); P.pooled = static_cast<__nv_bfloat16*>(pooled);
  P.bn = bn; P.delta = delta; P.counters = counters; P.eps = eps; P.relu = relu; P.k_pad = k_pad;
  P.h = h; P.w2 = w / 2 * 3; P.ho = (h - 1) / 2 + 1; P.wo = (w - 1) / 2 + 1;
  P.hp = (P.ho - 1) / 2 + 1; P.wp = (P.wo - 1) / 2 + 1;
  P.col_tiles = (P.wp + kCols - 1) / kCols;
  if (plan->n != n || plan->h != h || plan->w != w) {
    if (cudaDeviceGetAttribute(&plan->sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || plan->sms <= 0) plan->sms = 148;
    split_strips((long long)n * P.col_tiles, P.hp, plan);
    plan->n = n; plan->h = h; plan->w = w;
  }
  const int sms = plan->sms;
  P.segs = plan->segs; P.per = plan->per;
  const long long strips = (long long)n * P.col_tiles * P.segs;
  if (w % 2 || strips > 0x3fffffffll) return (int)cudaErrorInvalidValue;
  P.strips = (int)strips;
  P.items = (P.strips + 1) / 2;
  static bool set[64] = {};
  if (!set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(stem_pool_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return (int)e;
    set[dev] = true;
  }
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = stream;
  cfg.gridDim = dim3((unsigned)(P.items < sms ? P.items : sms), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = 227 * 1024;                   // (as the layer kernels: no reconfiguration between them)
  const cudaError_t e = cudaLaunchKernelEx(&cfg, stem_pool_kernel, P);
  return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}

}  // namespace cg
