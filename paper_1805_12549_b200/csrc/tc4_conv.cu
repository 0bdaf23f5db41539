// Channel-gated convolution on tcgen05 tensor cores: the window kernel (bf16 and int8).
//
// D[pixel, channel] = sum over taps and channels, N = 64 or 128 output channels.  Two things bound the other
// layer kernels on most shapes: rows of a tile spent on padding, and a chain of small copies per job.  Here
// one im2col-mode TMA copy brings everything a job needs of an input-channel chunk, and jobs are any
// consecutive pixels:
//   window mode (3x3, stride 1)  the bounding box of the im2col map has w + 1 columns and h + 1 rows per
//       image, so a run of consecutive positions is the batch stacked with its zero padding (neighbouring
//       rows and images share it).  Output pixel (h, w) of image n is position (n*(h+1) + h)*(w+1) + w, and
//       its filter tap (r, s) is the position r*(w+1) + s further on: a patch of 128 + 2*(w+2) positions
//       serves all nine taps, each as another start row of the same shared-memory operand.  Positions in the
//       padding are computed and dropped: (w/(w+1))*(h/(h+1)) of the rows are pixels, whatever the image size.
//   stride-2 windows (pairs, even extents)  the pixels of odd or even rows and columns are four lattices of pitch
//       w' + 1 and h' + 1, and a window over each serves four, two, two or one of the taps.  The taps come in the order 0..8 all
//       the same, so that all four patches of a chunk are there at a time: in the order 0 2 6 8 1 7 3 5 4, which needs one, a
//       gate whose partial sum lies within an fp32 rounding of its threshold could decide otherwise than tap by tap.  (int8 sums
//       have no rounding: they take that order where the weights leave no room.)  bf16 layers whose weights leave no room have a
//       patch per filter row: of its two lattices the odd columns serve the first and last tap, the even ones the middle tap.
//   tap mode (other strides, wide images)  one copy per filter tap and chunk, of 128 output pixels; no row is
//       dropped.  1x1 layers of any stride: one copy per chunk.
// The partial sum P and the conditional sum R have separate TMEM accumulators, two (N = 128) or four
// (N = 64) jobs deep, and both are computed for every pixel: a block of 128 pixels and 64 channels always
// holds a firing gate at the densities in use, and waiting for the gate costs more than it saves.  So the
// K loop is one run of MMAs per job and the epilogue one pass: d = (P >= t), y = f(BN1(P)) or f(BN2(P+R)).
// Pairs look at the thresholds, though: the jobs of a column tile in which no gate can fire run the base rows only
// (run_roles<BASE>; all thresholds +inf, us for all rows and for the base rows: 512@4x4 b256 28 and 14.6, 256@14x14 b64
// 18.3 and 13.2, 512@7x7 b64 18.0 and 11.7).  That is a second copy of the role code, chosen by a look that a warp
// takes while the block sets up: with row tables and bounds as variables of one copy, and a function call in its
// epilogue, every layer took 0.5 to 1.5 us more.
//
// Jobs are 256 pixels of a CTA pair (cta_group::2): each SM holds half of a job's pixels and half of its
// weights, which halves what an SM has to fetch from L2 and what an MMA reads of shared memory (one CTA's
// 128 x 128 MMA takes the whole 128 bytes per clock).  Layers of few jobs with long K loops (tc4_plan has
// the lines) instead split the K loop of a 128-pixel job over the 2, 4 or 8 CTAs of a cluster: every CTA finishes 1/split of the rows, and is sent the
// others' sums of those by bulk copies between the CTAs' shared memories.
//
// Warp roles (640 threads): 0 = patch producer, 2 = weight producer, 1 = MMA issuer, 4-19 = epilogue (TMEM
// lane quadrant x 32 channels).  The epilogue keeps out of shared memory, whose bandwidth the MMAs' operands
// take: it reads TMEM in the fragment layout, keeps the constants of its channels in registers and writes
// 16-byte pieces, four lanes to a 64-byte run.  The K loop goes by filter rows (three taps, up to 12 MMAs, one weight
// stage), written out for the kinds of rows a layer has (issue_jobs): a row then costs its issuer 170 cycles beside its MMAs.
// As a table of row kinds it took 570 to 1,000, two issuers in turns, more than the MMAs: 128@16x16 b256 23.6 us for 20.0
// now, 128@28x28 b128 31.8 for 26.1, 64@56x56 b128 37.8 for 35.2 (graphs of 20 calls).  The copies of a pair's second CTA
// count on its leader's barriers without an arrival of their own: with one per slot, and copies issued from divergent
// code, every streamed layer waited for its weights (512 channels, 4x4, batch 256: 67 us).
//
// Measured (graphs of 20 calls, us; in brackets with two issuers that walked a table, before the steps that the comments
// below describe): 128@16x16 b256 17.4 (23.0), 256@8x8 b256 20.4 (23.7), 512@4x4 b256 23.8 (27.8), 64@56x56 b64 with residual
// 22.4 (23.4), b128 39 (43), 128->256 stride 2 at 28x28 b64 13.6 (16.0), int8 128@28x28 b64 15.8 (17.6), 128@28x28 b128 22.8 (30.7),
// 64->128 stride 2 b128 18.5 (26.4); one image: 64@56x56 5.9 (7.4), 512@7x7 7.3 (8.1).  What bounds it now: 256 and 512
// channels their MMAs in whole rounds of jobs (9,000 cycles a job of 256 channels, 9,200 of MMAs); 128 channels the same behind a
// start of 4,000 cycles and a tail of 4,000; 64 channels operand reads, 2,100 cycles a job of 1,550 of MMAs at 43 each beside
// the patches' writes to shared memory; int8 its epilogue; one image the chain of first copies (2,500 cycles), MMAs, exchange
// and epilogue.  Neither a fixed order of first copies (patch, weights, patches) nor two small CTAs to an SM made it faster.
// Every mbarrier wait is bounded; on expiry the CTA records CG_ERR_DEVICE_TIMEOUT with the id of the wait
// and leaves.
#include <cstring>
#include <type_traits>

#include "direct_point.cuh"
#include "ptx.cuh"
#include "tc4_conv.cuh"

namespace cg {

namespace {

constexpr int kT4Threads = 640;
constexpr int kEpiWarp0 = 4, kEpiWarps = 16, kEpiThreads = kEpiWarps * 32;
constexpr unsigned kSumPitch = (64 + 4) * 4;           // a row of partial sums on its way to the CTA that finishes it
constexpr int kMaxNA = 8, kMaxNB = 16;
constexpr int kSpinLimit = 1 << 21;
constexpr long long kWaitCycles = 2000000000ll;
constexpr unsigned kOffConsts = 1024;                  // behind the barriers; 32 bytes per channel
constexpr unsigned kOffRows = kOffConsts + 128 * 32;   // the row table
constexpr unsigned kOffStages = 6 * 1024;              // weight stages, then patch slots
static_assert(kOffRows + kTc4MaxRows * sizeof(Tc4Row) <= kOffStages, "row table");
constexpr unsigned kSmemBytes = 227 * 1024;

struct Tc4Params {
  LayerDims L;
  cg_bn_params bn;
  const float* delta;
  const __nv_bfloat16* residual;
  void* y;
  uint32_t* mask;
  unsigned long long* counters;
  const __nv_bfloat16 *x, *w_cond;   // (read by infinite_sums only)
  Tc4Plan P;
};

// The weights' tensor maps; HALF: a layer whose last round is in halves (Tc4Plan::half_job) has maps for those, too.  (An
// instance of the kernel of its own: the choice between the maps, operand starts and instruction descriptors costs others 1 to 5 %.)
template <bool HALF> struct WeightMaps { CUtensorMap wb, wc; };
template <> struct WeightMaps<true> { CUtensorMap wb, wc, half_wb, half_wc; };

// Rows of a cluster's job that each of its CTAs finishes: the positions that there are, in even shares.
__device__ __forceinline__ int split_rows(const Tc4Plan& P, int group) {
  const int there = min(128, P.positions - group * 128);
  return ((there + P.split - 1) / P.split + 1) & ~1;
}

struct Shared4 {
  uint64_t a_full[kMaxNA], a_empty[kMaxNA];
  uint64_t b_full[kMaxNB], b_empty[kMaxNB];
  uint64_t acc_full[4], acc_empty[4];
  uint64_t sums;         // the cluster's sums of this CTA's rows have arrived
  uint32_t tmem_base;
  uint32_t abort_flag;
  uint32_t active, rows_active;
  uint32_t epi_done;     // epilogue warps that have added theirs
  uint32_t maybe_shut;   // no gate of the column tile could fire when the block started
};
static_assert(sizeof(Shared4) <= kOffConsts, "barrier block");

__device__ __noinline__ bool wait4_slow(Shared4* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity,
                                        int site) {
  const long long t0 = clock64();
  for (int i = 0; i < kSpinLimit; ++i) {
    if (ptx::mbar_try_wait(bar, parity)) return true;
    if ((i & 15) == 15) {
      if (*(volatile uint32_t*)&sh->abort_flag) return false;
      if (clock64() - t0 > kWaitCycles) break;
    }
  }
  if (atomicCAS(&counters[CNT_STATUS], 0ull, (unsigned long long)CG_ERR_DEVICE_TIMEOUT) == 0ull)
    atomicExch(&counters[CNT_SITE], (unsigned long long)(400 + site));
  atomicExch(&sh->abort_flag, 1u);
  return false;
}

// Taken by one lane.
__device__ __forceinline__ bool wait4_one(Shared4* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity,
                                          int site) {
  if (ptx::mbar_try_wait(bar, parity, 0u)) return true;
  return wait4_slow(sh, counters, bar, parity, site);
}

// Taken by every lane of a convergent warp; the outcome is warp-uniform.
__device__ __forceinline__ bool wait4(Shared4* sh, unsigned long long* counters, uint64_t* bar, uint32_t parity,
                                      int site) {
  bool ok = ptx::mbar_try_wait(bar, parity, 0u);
  if (!__all_sync(0xffffffffu, ok)) ok = __all_sync(0xffffffffu, wait4_slow(sh, counters, bar, parity, site));
  return ok;
}

// A ring position: slot and the phase parity of its "full" barrier.
struct Cursor {
  int slot;
  uint32_t par;
  __device__ __forceinline__ void next(int n) { if (++slot == n) { slot = 0; par ^= 1u; } }
};

// The MMAs of one row of the table: up to three tiles of NKS K slices.
template <bool PAIR, bool I8, int NKS>
__device__ __forceinline__ void issue_row(int tiles, uint32_t d, uint32_t hi, uint32_t a, uint32_t a_step, uint32_t b0,
                                          uint32_t b1, uint32_t b2, uint32_t idesc, uint32_t acc) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    if (s >= tiles) break;
    const uint32_t a_s = a + (uint32_t)s * a_step, b_s = s == 0 ? b0 : s == 1 ? b1 : b2;
#pragma unroll
    for (int k = 0; k < NKS; ++k)
      ptx::umma<PAIR, I8>(d, ((uint64_t)hi << 32) | (a_s + 2u * k), ((uint64_t)hi << 32) | (b_s + 2u * k), idesc,
                          s == 0 && k == 0 ? acc : 1u);
  }
}

// From a filter row's first tap to its tap s, in 16-byte units of the patch: `step` each, or, for kTwoPatches (a patch per
// filter row at stride 2), the odd columns' next position (s = 2) and the patch of the even columns behind them (s = 1).
constexpr int kLatticeSlots = 8;                              // patches of a lattice at most, where weights stream
constexpr int kLatticeRows = 136;                              // positions per patch: 129, in whole swizzle atoms
constexpr uint32_t kTwoPatches = ~0u;
__device__ __forceinline__ uint32_t tap_step(uint32_t s, uint32_t step) {
  return step != kTwoPatches ? s * step : s == 1 ? kLatticeRows * 8u : s * 4u;
}

// The taps [T0, T1) of a chunk, K slices [K0, K0 + NK) of each: PER taps of NK slices share a weight tile, B0 is the first
// tile of the stage.  Tap t reads the patch at (t / 3 - R0) * row_lo + tap_step(t % 3).
template <bool PAIR, bool I8, int T0, int T1, int R0, int K0, int NK, int PER, int B0>
__device__ __forceinline__ void issue_taps(uint32_t d, uint32_t hi, uint32_t a, uint32_t row_lo, uint32_t step, uint32_t b,
                                           uint32_t tile, uint32_t idesc, uint32_t acc) {
#pragma unroll
  for (int t = T0; t < T1; ++t) {
    const uint32_t a_t = a + (uint32_t)(t / 3 - R0) * row_lo + tap_step((uint32_t)(t % 3), step) + 2u * K0;
    const uint32_t b_t = b + (uint32_t)(t / PER - B0) * tile + (uint32_t)((t % PER) * NK) * 2u;
#pragma unroll
    for (int k = 0; k < NK; ++k)
      ptx::umma<PAIR, I8>(d, ((uint64_t)hi << 32) | (a_t + 2u * k), ((uint64_t)hi << 32) | (b_t + 2u * k), idesc,
                          t == T0 && k == 0 ? acc : 1u);
  }
}

// The same with the weights' K slices packed (Tc4Plan::packed): a tap has PT conditional slices, of which the patch's chunk takes
// NK from FIRST on, beside its own slices from K0 on.  Filter row R; `a` is its first tap.
template <bool I8, int R, int PT, int FIRST, int K0, int NK>
__device__ __forceinline__ void issue_packed(uint32_t d, uint32_t hi, uint32_t a, uint32_t step, uint32_t b, uint32_t tile, uint32_t idesc,
                                             uint32_t acc) {
#pragma unroll
  for (int t = 0; t < 3; ++t)
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      const int s = (3 * R + t) * PT + FIRST + k;
      ptx::umma<true, I8>(d, ((uint64_t)hi << 32) | (a + tap_step((uint32_t)t, step) + 2u * (K0 + k)),
                          ((uint64_t)hi << 32) | (b + (uint32_t)(s / 4) * tile + (uint32_t)(s % 4) * 2u), idesc, t == 0 && k == 0 ? acc : 1u);
    }
}

// Stride-2 windows: patch of tap t (bit 0: even columns, bit 1: even rows), the taps in the order of the sums or (BY_PATCH) by
// patches, and in which places of that order a patch is taken first and last.
__host__ __device__ constexpr int lattice_of(int t) { return (t / 3 == 1 ? 2 : 0) + (t % 3 == 1 ? 1 : 0); }
template <bool BY_PATCH> __host__ __device__ constexpr int lattice_tap(int i) { return BY_PATCH ? (int)((0x453718620ull >> (4 * i)) & 15) : i; }
template <bool BY_PATCH> __host__ __device__ constexpr bool lattice_first(int i) {
  for (int k = 0; k < i; ++k)
    if (lattice_of(lattice_tap<BY_PATCH>(k)) == lattice_of(lattice_tap<BY_PATCH>(i))) return false;
  return true;
}
template <bool BY_PATCH> __host__ __device__ constexpr bool lattice_last(int i) {
  for (int k = i + 1; k < 9; ++k)
    if (lattice_of(lattice_tap<BY_PATCH>(k)) == lattice_of(lattice_tap<BY_PATCH>(i))) return false;
  return true;
}
// Tap t of such a patch: NK slices from K0 on.  Its weights: PT slices a tap from FIRST on, packed (PT > 0), or tile t % 3 of a stage.
template <bool I8, int PT, int FIRST, int K0, int NK>
__device__ __forceinline__ void issue_lattice_tap(int t, uint32_t d, uint32_t hi, uint32_t a, uint32_t row_lo, uint32_t b, uint32_t tile,
                                                  uint32_t idesc, uint32_t acc) {
  const uint32_t a_t = a + (t / 3 == 2 ? row_lo : 0u) + (t % 3 == 2 ? 8u : 0u);
#pragma unroll
  for (int k = 0; k < NK; ++k) {
    const int s = t * PT + FIRST + k;
    const uint32_t b_t = PT > 0 ? b + (uint32_t)(s / 4) * tile + (uint32_t)(s % 4) * 2u : b + (uint32_t)(t % 3) * tile + 2u * k;
    ptx::umma<true, I8>(d, ((uint64_t)hi << 32) | (a_t + 2u * (K0 + k)), ((uint64_t)hi << 32) | b_t, idesc, k == 0 ? acc : 1u);
  }
}

// One row of the table in shared memory.
__device__ __forceinline__ Tc4Row row_at(uint32_t table, int i) {
  const uint4 v = ptx::ld_shared_16(table + (uint32_t)i * 16u);
  Tc4Row r;
  r.a_off = (uint16_t)v.x; r.b_off[0] = (uint16_t)(v.x >> 16); r.b_off[1] = (uint16_t)v.y; r.b_off[2] = (uint16_t)(v.y >> 16);
  r.bx = (uint16_t)v.z; r.bstep = (uint16_t)(v.z >> 16);
  r.flags = (uint8_t)v.w; r.kind = (uint8_t)(v.w >> 8); r.chunk = (uint8_t)(v.w >> 16); r.tap_row = (uint8_t)(v.w >> 24);
  return r;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// max(v, 0) of two bf16 values; a NaN gives 0
__device__ __forceinline__ uint32_t relu_bf16x2(uint32_t v) {
  const uint32_t zero = 0u;
  const __nv_bfloat162 h = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&v), *reinterpret_cast<const __nv_bfloat162*>(&zero));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// int8 layers: requantised in 64-bit integers, rounded half up (the half is in `off`: add_half), clamped to 32 bits.
__device__ __forceinline__ long long add_half(long long off, int shift) { return (long long)((unsigned long long)off + (1ull << (shift - 1))); }
__device__ __forceinline__ int requantise(int mul, long long off, int acc, int shift) {
  const long long z = (long long)((unsigned long long)((long long)acc * mul) + (unsigned long long)off);
  const int top = (int)(z >> 32), lo = (int)__funnelshift_r((uint32_t)z, (uint32_t)top, (uint32_t)shift);
  return (top >> shift) == (lo >> 31) ? lo : (top >> 31) ^ 0x7fffffff;
}
// Four of them, clamped to [lo, 127], as bytes.
__device__ __forceinline__ uint32_t pack_s8(const int* v, int lo) {
  uint32_t d;
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, 0;" : "=r"(d) : "r"(max(v[3], lo)), "r"(max(v[2], lo)));
  asm("cvt.pack.sat.s8.s32.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(max(v[1], lo)), "r"(max(v[0], lo)), "r"(d));
  return d;
}

// Whether no gate of the column tile can fire: thresholds of +inf (or not a number); int8: beyond every sum.  (Finite
// thresholds that no partial sum happens to reach are not looked for: the conditional rows would have to wait for the
// base rows and the epilogue.)  Taken by a whole warp; reads past L1, so that it may run before the kernels in front
// of this one are done.
template <int NT, bool I8>
__device__ __forceinline__ bool gates_shut(const Tc4Params& prm, int tile_n, int lane) {
  bool open = false;
#pragma unroll
  for (int c = 0; c < NT; c += 32) {
    const int ch = tile_n * NT + c + lane;
    if (ch >= prm.L.c_out) continue;
    if (I8) open = open || __ldcg(prm.bn.q_gate_thr + ch) <= prm.L.kh * prm.L.kw * prm.L.c_p * (128 * 128);
    else open = open || __ldcg(prm.delta + ch) < __int_as_float(0x7f800000);
  }
  return !__any_sync(0xffffffffu, open);
}

// A tie fires, at +inf too: outputs whose partial sum of +inf meets a threshold of +inf, in a column tile without
// conditional rows.  Lane by row (pixel m, or -1), 32 channels from ch on: R comes from its definition.
__device__ __forceinline__ void infinite_sums(const Tc4Params& prm, uint32_t t_col, const float* t, const float* t2,
                                           const float4* k, int ch, int m) {
  const LayerDims& L = prm.L;
  const int row = m / L.wo, n = row / L.ho;
#pragma unroll 1
  for (int col = 0; col < 32; ++col) {
    uint32_t v;
    __syncwarp();                                              // (also orders the lanes' stores to y)
    ptx::tmem_ld1(t_col + (uint32_t)col, v);
    const float p = __uint_as_float(v);
    const int c = 8 * ((col >> 1) & 3) + 2 * (col >> 3) + (col & 1);   // (the weight tiles' row order)
    if (m < 0 || !(p >= t[c]) || !(p <= t2[c])) continue;
    const float sum = p + conv_point<__nv_bfloat16>(L, prm.x, prm.w_cond, n, row - n * L.ho, m - row * L.wo, ch + c, L.c_p, L.c_r);
    const long long at = (long long)m * L.c_out + ch + c;
    float o = fmaf(k[c].z, sum, k[c].w);
    if (prm.residual) o += __bfloat162float(prm.residual[at]);
    if (L.relu) o = fmaxf(o, 0.f);
    ((__nv_bfloat16*)prm.y)[at] = __float2bfloat16_rn(o);
  }
  __syncwarp();
}

// A ring of slots as the issuer walks it: operand address (16-byte units) and the phase parity of the "full" barrier.
struct IssueRing {
  int slot;
  uint32_t par, at;
  __device__ __forceinline__ void next(int n, uint32_t size, uint32_t first) {
    at += size;
    if (++slot == n) { slot = 0; par ^= 1u; at = first; }
  }
};

// The MMAs of all jobs of a pair, taken by one lane of its first CTA.  MODE and KP (slices of the first chunk that belong to
// the base path; 4: the base path is whole chunks) are constants, so that a filter row is one look at its weights' barrier,
// its MMAs and a commit: walked from a table of row kinds, a row's loads, tests and branches took 700 cycles beside the 576 of
// nine MMAs of 64, two issuers taking turns.
// CH: chunks of a layer with packed weights, else 0.
template <int NT, bool I8, bool BASE, bool HALF, int MODE, int KP, int CH = 0>
__device__ __forceinline__ void issue_jobs(const Tc4Params& prm, Shared4* sh, uint32_t a0, uint32_t b0, uint32_t tmem, int group,
                                           int jobs) {
  constexpr int kAcc = 512 / (2 * NT);
  constexpr uint32_t kTileU = (uint32_t)(NT / 2) * 8u;         // a weight tile, 16-byte units
  constexpr bool kWin = MODE == kTc4Window;
  const Tc4Plan& P = prm.P;
  uint32_t idesc = I8 ? ptx::idesc_s8(256, NT) : ptx::idesc_bf16(256, NT);
  const uint32_t hi = (uint32_t)(ptx::smem_desc(0, 1024, 2) >> 32);
  const uint32_t a_size = (uint32_t)P.slot_bytes >> 4, b_size = (uint32_t)P.stage_bytes >> 4;
  const uint32_t row_lo = kWin || MODE == kTc4Lattice ? (uint32_t)P.wp * 8u : 0u;
  constexpr uint32_t kStep = kWin ? 8u : MODE == kTc4Rows2 ? kTwoPatches : 1024u;   // from tap to tap of a filter row
  const int na = P.na, nb = P.nb;
  const bool resident = P.resident != 0;
  const int ck = I8 ? 128 : 64;
  const int chunks = BASE ? (prm.L.c_p + ck - 1) / ck : prm.L.c_in / ck, base_chunks = KP == 4 ? prm.L.c_p / ck : 0;
  IssueRing a{0, 0u, a0}, b{0, 0u, b0};
  bool ok = true, a_seen = false, b_seen = false;
  int tiles_seen = 0;                                          // (packed weights)
  bool new_b = true;                                           // weights are waited for (resident ones: by the first job)
  uint32_t a_at = 0, b_at = 0;
  int a_slot = 0, b_slot = 0;
  auto take_a = [&]() {
    if (!a_seen) ok = ok && wait4_one(sh, prm.counters, &sh->a_full[a.slot], a.par, 4);
    a_at = a.at; a_slot = a.slot;
    a.next(na, a_size, a0);
    a_seen = false;
  };
  auto take_b = [&]() {
    if (new_b && !b_seen) ok = ok && wait4_one(sh, prm.counters, &sh->b_full[b.slot], b.par, 5);
    b_at = b.at; b_slot = b.slot;
    b.next(nb, b_size, b0);
    // a look at the next stage's barrier, whose answer arrives while this one's MMAs are issued
    b_seen = new_b && ptx::mbar_test_wait(&sh->b_full[b.slot], b.par);
  };
  auto need_tile = [&](int tile) {
    for (; ok && tiles_seen <= tile; tiles_seen += 3)
      ok = wait4_one(sh, prm.counters, &sh->b_full[tiles_seen / 3], 0, 5);
  };
  auto look_a = [&]() { a_seen = ptx::mbar_test_wait(&sh->a_full[a.slot], a.par); };
  auto free_a = [&]() { ptx::umma_commit_pair(&sh->a_empty[a_slot]); };
  auto free_b = [&](int slot) { if (!resident) ptx::umma_commit_pair(&sh->b_empty[slot]); };
  for (int j = 0; j < jobs; ++j) {
    const int stage = j % kAcc;
    ok = wait4_one(sh, prm.counters, &sh->acc_empty[stage], ((j / kAcc) & 1) ^ 1, 3);
    if (!ok) return;
    ptx::tc_fence_after();
    const uint32_t d_p = tmem + (uint32_t)(stage * 2 * NT), d_r = d_p + NT;
    if (HALF && j == P.half_job) {                             // 64 of the columns: half of the rows of every weight tile
      idesc = I8 ? ptx::idesc_s8(256, 64) : ptx::idesc_bf16(256, 64);
      if (resident) b0 += (uint32_t)(group & 1) * (kTileU / 2u);
    }
    if (resident) { b = IssueRing{0, 0u, b0}; new_b = j == 0; b_seen = false; }
    if constexpr (MODE == kTc4Lattice) {
      // four patches a chunk; packed weights (CH > 0) or a stage per filter row
      constexpr bool kByPatch = I8 && CH == 2;
      constexpr int KB = CH > 0 ? KP : 4, PT = CH > 0 ? 4 * CH - KP : 0;
      const uint32_t bc = b0 + (uint32_t)P.tiles_base * kTileU;
      auto chunk = [&](auto second, int q) {
        constexpr int Q = decltype(second)::value, FIRST = Q ? 4 - KB : 0, K0 = Q ? 0 : KB, NK = Q ? 4 : 4 - KB;
        uint32_t at[4] = {0u, 0u, 0u, 0u};
        int slot[4] = {0, 0, 0, 0};
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          const int t = lattice_tap<kByPatch>(i), p = lattice_of(t);
          if (lattice_first<kByPatch>(i)) { take_a(); at[p] = a_at; slot[p] = a_slot; }
          if (CH == 0 && t % 3 == 0) take_b();
          if (CH > 0 && Q == 0) need_tile((t * KB + KB - 1) / 4);
          if (CH > 0 && !BASE) need_tile(P.tiles_base + (t * PT + FIRST + NK - 1) / 4);
          if (!ok) return;
          if (i < 8 && lattice_first<kByPatch>(i + 1)) look_a();
          if (CH == 0) {
            issue_lattice_tap<I8, 0, 0, 0, 4>(t, q < base_chunks ? d_p : d_r, hi, at[p], row_lo, b_at, kTileU, idesc,
                                              i == 0 && (q == 0 || q == base_chunks) ? 0u : 1u);
          } else {
            if (Q == 0) issue_lattice_tap<I8, KB, 0, 0, KB>(t, d_p, hi, at[p], row_lo, b0, kTileU, idesc, i ? 1u : 0u);
            if (!BASE) issue_lattice_tap<I8, PT, FIRST, K0, NK>(t, d_r, hi, at[p], row_lo, bc, kTileU, idesc, Q || i ? 1u : 0u);
          }
          if (lattice_last<kByPatch>(i)) ptx::umma_commit_pair(&sh->a_empty[slot[p]]);
          if (CH == 0 && t % 3 == 2) free_b(b_slot);
        }
      };
      if constexpr (CH > 0) {
        chunk(std::integral_constant<int, 0>{}, 0);
        if (ok && CH == 2 && !BASE) chunk(std::integral_constant<int, 1>{}, 1);
      } else {
#pragma unroll 1
        for (int q = 0; q < chunks && ok; ++q) chunk(std::integral_constant<int, 0>{}, q);
      }
      if (!ok) return;
    } else if constexpr (MODE == kTc4Rows2 && CH > 0) {
      // a patch per chunk and filter row
      constexpr int PT = 4 * CH - KP;                          // conditional slices of a tap
      const uint32_t bc = b0 + (uint32_t)P.tiles_base * kTileU;
      auto filter_row = [&](auto chunk, auto row) {
        constexpr int Q = decltype(chunk)::value, R = decltype(row)::value, FIRST = Q ? 4 - KP : 0, K0 = Q ? 0 : KP, NK = Q ? 4 : 4 - KP;
        take_a();
        need_tile(BASE ? ((3 * R + 3) * KP - 1) / 4 : P.tiles_base + ((3 * R + 2) * PT + FIRST + NK - 1) / 4);
        if (!ok) return;
        look_a();
        if (Q == 0) issue_taps<true, I8, 3 * R, 3 * R + 3, R, 0, KP, 4 / KP, 0>(d_p, hi, a_at, 0, kStep, b0, kTileU, idesc, R ? 1u : 0u);
        if (!BASE) issue_packed<I8, R, PT, FIRST, K0, NK>(d_r, hi, a_at, kStep, bc, kTileU, idesc, Q || R ? 1u : 0u);
        free_a();
      };
      auto chunk = [&](auto q) {
        filter_row(q, std::integral_constant<int, 0>{});
        if (ok) filter_row(q, std::integral_constant<int, 1>{});
        if (ok) filter_row(q, std::integral_constant<int, 2>{});
      };
      chunk(std::integral_constant<int, 0>{});
      if (ok && CH == 2 && !BASE) chunk(std::integral_constant<int, 1>{});
      if (!ok) return;
    } else if constexpr (CH > 0) {
      static_assert(CH == 0 || CH == 2, "two chunks");
      constexpr int PT = 8 - KP;                               // conditional slices of a tap
      const uint32_t bc = b0 + (uint32_t)P.tiles_base * kTileU;
      take_a();
      need_tile(P.tiles_base - 1);
      if (!ok) return;
      issue_taps<true, I8, 0, 9, 0, 0, KP, 4 / KP, 0>(d_p, hi, a_at, row_lo, kStep, b0, kTileU, idesc, 0u);
      if (!BASE) {
        auto upto = [&](int last) { need_tile(P.tiles_base + last / 4); return ok; };
        if (!upto(2 * PT + 3 - KP)) return;
        issue_packed<I8, 0, PT, 0, KP, 4 - KP>(d_r, hi, a_at, kStep, bc, kTileU, idesc, 0u);
        if (!upto(5 * PT + 3 - KP)) return;
        issue_packed<I8, 1, PT, 0, KP, 4 - KP>(d_r, hi, a_at + row_lo, kStep, bc, kTileU, idesc, 1u);
        if (!upto(8 * PT + 3 - KP)) return;
        look_a();
        issue_packed<I8, 2, PT, 0, KP, 4 - KP>(d_r, hi, a_at + 2u * row_lo, kStep, bc, kTileU, idesc, 1u);
        free_a();
        take_a();
        if (!upto(9 * PT - 1)) return;
        issue_packed<I8, 0, PT, 4 - KP, 0, 4>(d_r, hi, a_at, kStep, bc, kTileU, idesc, 1u);
        issue_packed<I8, 1, PT, 4 - KP, 0, 4>(d_r, hi, a_at + row_lo, kStep, bc, kTileU, idesc, 1u);
        look_a();
        issue_packed<I8, 2, PT, 4 - KP, 0, 4>(d_r, hi, a_at + 2u * row_lo, kStep, bc, kTileU, idesc, 1u);
      }
      free_a();
    } else for (int q = 0; q < chunks; ++q) {
      if constexpr (MODE == kTc4Chunks) {
        // up to three chunks of a 1x1 layer per slot
        take_a(); take_b();
        if (!ok) return;
        look_a();
        const int tiles = chunks - q < 3 ? chunks - q : 3;
        const uint32_t acc = q ? 1u : 0u;
        issue_taps<true, I8, 0, 1, 0, 0, 4, 1, 0>(d_p, hi, a_at, 0, kStep, b_at, kTileU, idesc, acc);
        if (tiles > 1) issue_taps<true, I8, 1, 2, 0, 0, 4, 1, 0>(d_p, hi, a_at, 0, kStep, b_at, kTileU, idesc, 1u);
        if (tiles > 2) issue_taps<true, I8, 2, 3, 0, 0, 4, 1, 0>(d_p, hi, a_at, 0, kStep, b_at, kTileU, idesc, 1u);
        q += 2;
        free_b(b_slot);
        free_a();
      } else if (KP < 4 && q == 0) {
        // the first chunk holds the base channels (KP slices of every tap, several taps per weight tile) and the first
        // conditional ones
        constexpr int kCond = 4 - KP > 0 ? 4 - KP : 1, kFirst = KP < 4 ? KP : 0;
        if (kWin) take_a();
        take_b();
        const uint32_t base_at = b_at;
        const int base_slot = b_slot;
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          if (!kWin) take_a();
          if (!ok) return;
          if (kWin) {
            if (r == 0) {
              if (KP == 1) issue_taps<true, I8, 0, 9, 0, 0, 1, 4, 0>(d_p, hi, a_at, row_lo, kStep, base_at, kTileU, idesc, 0u);
              else issue_taps<true, I8, 0, 6, 0, 0, 2, 2, 0>(d_p, hi, a_at, row_lo, kStep, base_at, kTileU, idesc, 0u);
              free_b(base_slot);
            }
          } else {
            if (KP == 1) {
              if (r == 0) issue_taps<true, I8, 0, 3, 0, 0, 1, 4, 0>(d_p, hi, a_at, 0, kStep, base_at, kTileU, idesc, 0u);
              if (r == 1) issue_taps<true, I8, 3, 6, 1, 0, 1, 4, 0>(d_p, hi, a_at, 0, kStep, base_at, kTileU, idesc, 1u);
              if (r == 2) issue_taps<true, I8, 6, 9, 2, 0, 1, 4, 0>(d_p, hi, a_at, 0, kStep, base_at, kTileU, idesc, 1u);
              if (r == 2) free_b(base_slot);
            } else {
              if (r == 0) issue_taps<true, I8, 0, 3, 0, 0, 2, 2, 0>(d_p, hi, a_at, 0, kStep, base_at, kTileU, idesc, 0u);
              if (r == 1) issue_taps<true, I8, 3, 6, 1, 0, 2, 2, 0>(d_p, hi, a_at, 0, kStep, base_at, kTileU, idesc, 1u);
              if (r == 1) free_b(base_slot);
            }
          }
          if (KP == 2 && r == 2) {                             // the last three taps have a stage of their own
            take_b();
            if (!ok) return;
            issue_taps<true, I8, 6, 9, kWin ? 0 : 2, 0, 2, 2, 3>(d_p, hi, a_at, row_lo, kStep, b_at, kTileU, idesc, 1u);
            free_b(b_slot);
          }
          if (!BASE) {
            take_b();
            if (!ok) return;
            if (!kWin || r == 2) look_a();
            issue_taps<true, I8, 0, 3, 0, kFirst, kCond, 1, 0>(d_r, hi, a_at + (uint32_t)r * row_lo, 0, kStep, b_at, kTileU,
                                                              idesc, r ? 1u : 0u);
            free_b(b_slot);
          }
          if (!kWin || r == 2) free_a();
        }
      } else {
        if (kWin) take_a();
        const uint32_t d = q < base_chunks ? d_p : d_r;
        uint32_t acc = q == 0 || (KP == 4 && q == base_chunks) ? 0u : 1u;
#pragma unroll 1
        for (int r = 0; r < 3; ++r) {
          if (!kWin) take_a();
          take_b();
          if (!ok) return;
          if (!kWin || r == 2) look_a();
          issue_taps<true, I8, 0, 3, 0, 0, 4, 1, 0>(d, hi, a_at, 0, kStep, b_at, kTileU, idesc, acc);
          acc = 1u;
          free_b(b_slot);
          if (!kWin) free_a();
          else a_at += row_lo;
        }
        if (kWin) free_a();
      }
    }
    ptx::umma_commit_pair(&sh->acc_full[stage]);
  }
}

// What the warps of a block do (see the top of the file).  BASE: the jobs of a column tile whose gates cannot fire, which run
// the base rows only.
template <int NT, bool I8, bool PAIR, bool HALF, bool BASE>
__device__ __forceinline__ void run_roles(const CUtensorMap& map_x, const WeightMaps<HALF>& maps, const Tc4Params& prm, uint8_t* smem, int warp, int lane, int part, int tile_n,
                                          int group, int groups, int jobs, uint32_t tmem) {
  constexpr bool SPLIT = !PAIR;
  const CUtensorMap &map_wb = maps.wb, &map_wc = maps.wc;
  const LayerDims& L = prm.L;
  const Tc4Plan& P = prm.P;
  Shared4* sh = (Shared4*)smem;
  float4* s_k = (float4*)(smem + kOffConsts);                  // {a1, b1, a2, b2}
  float* s_t = (float*)(smem + kOffConsts + NT * 16);
  float* s_t2 = s_t + NT;
  int4* s_q = (int4*)(smem + kOffConsts);                      // {threshold, base and full multiplier, -}
  longlong2* s_o = (longlong2*)(smem + kOffConsts + NT * 16);  // {base, full offset}
  uint8_t* s_b = smem + P.off_b;
  uint8_t* s_a = smem + P.off_a;
  constexpr int kAcc = 512 / (2 * NT);                         // accumulator pairs in TMEM
  constexpr int kTileRows = PAIR ? NT / 2 : NT;                // rows of a weight tile in this CTA
  constexpr uint32_t kTile = kTileRows * 128;
  const int lo = SPLIT ? P.lo[part] : 0, hi = BASE ? P.base_rows : SPLIT ? P.lo[part + 1] : P.rows;
  const bool has_cond = !BASE && L.c_r > 0;
  const uint32_t table = ptx::smem_u32(smem + kOffRows);
  // first position of this CTA in job j
  auto job_pos = [&](int j) {
    if (!PAIR) return group * 128;
    return ((HALF && j == P.half_job ? group >> 1 : group) + j * groups) * 256 + part * 128;
  };
  // address of the leader's copy of a barrier, for copies and arrivals
  auto leader = [&](uint64_t* bar) { return PAIR ? ptx::map_cluster(ptx::smem_u32(bar), 0) : ptx::smem_u32(bar); };
  // (a pair's leader announces both CTAs' bytes; the other CTA's copies count on the leader's barrier: an
  // arrival of its own there costs it hundreds of cycles per slot)
  auto expect = [&](uint64_t* bar, uint32_t bytes) {
    if (!PAIR || part == 0) ptx::mbar_expect_tx(bar, PAIR ? 2u * bytes : bytes);
  };

  if (warp == 0) {
    // ============================================================ patch producer
    // (as everywhere in the role loops, the barrier of the next slot is looked at before the copies of this
    // one are issued: the answer arrives meanwhile)
    if (ptx::elect_one()) {
      Cursor c{0, 0};
      bool ok = true, seen = false;
      const int ip = P.wp * P.hp, st = P.mode == kTc4Window ? 1 : L.stride;
      for (int j = 0; j < jobs && ok; ++j) {
        const int pos = job_pos(j);
        const int n0 = pos / ip, rem = pos - n0 * ip, h0 = rem / P.wp, w0 = rem - h0 * P.wp;
        const int pos1 = pos + P.patch_rows;                   // start of a window's second load
        const int n1 = pos1 / ip, rem1 = pos1 - n1 * ip, h1 = rem1 / P.wp, w1 = rem1 - h1 * P.wp;
        if (PAIR && P.mode == kTc4Lattice) {
          // the patches of a chunk in the order in which they are taken: odd or even rows and columns
          const int ck = I8 ? 128 : 64, patches = 4 * (BASE ? (L.c_p + ck - 1) / ck : L.c_in / ck);
          for (int i = 0; i < patches && ok; ++i) {
            if (!seen) ok = wait4_one(sh, prm.counters, &sh->a_empty[c.slot], c.par ^ 1u, 1);
            if (!ok) break;
            uint8_t* dst = s_a + (size_t)c.slot * P.slot_bytes;
            uint64_t* full = &sh->a_full[c.slot];
            c.next(P.na);
            seen = ptx::mbar_test_wait(&sh->a_empty[c.slot], c.par ^ 1u);
            const uint32_t bar = leader(full);
            expect(full, (uint32_t)P.patch_rows * 128u);
            ptx::tma_load_im2col_4d<PAIR>(dst, &map_x, bar, (i >> 2) * ck, w0 * 2 - 1, h0 * 2 - 1, n0, (uint16_t)(i & 1),
                                          (uint16_t)((i >> 1) & 1));
          }
          continue;
        }
        Tc4Row next = row_at(table, lo);
        for (int i = lo; i < hi; ++i) {
          const Tc4Row s = next;
          if (i + 1 < hi) next = row_at(table, i + 1);
          if (!(s.flags & kRowANew)) continue;
          if (!seen) ok = wait4_one(sh, prm.counters, &sh->a_empty[c.slot], c.par ^ 1u, 1);
          if (!ok) break;
          uint8_t* dst = s_a + (size_t)c.slot * P.slot_bytes;
          uint64_t* full = &sh->a_full[c.slot];
          c.next(P.na);
          seen = ptx::mbar_test_wait(&sh->a_empty[c.slot], c.par ^ 1u);
          const uint32_t bar = leader(full);
          const int ch = (int)s.chunk * (I8 ? 128 : 64);
          const int tiles = P.mode == kTc4Window || P.mode == kTc4Rows2 ? P.loads : ((s.kind >> 4) & 3) + 1;
          expect(full, (uint32_t)(tiles * P.patch_rows) * 128u);
          if (P.mode == kTc4Window) {
            ptx::tma_load_im2col_4d<PAIR>(dst, &map_x, bar, ch, w0 - L.pad, h0 - L.pad, n0, 0, 0);
            if (tiles == 2)
              ptx::tma_load_im2col_4d<PAIR>(dst + (size_t)P.patch_rows * 128, &map_x, bar, ch, w1 - L.pad, h1 - L.pad, n1, 0, 0);
          } else if (P.mode == kTc4Rows2) {
            for (int k = 0; k < 2; ++k)
              ptx::tma_load_im2col_4d<PAIR>(dst + k * kLatticeRows * 128, &map_x, bar, ch, w0 * 2 - 1, h0 * 2 - 1, n0, (uint16_t)k,
                                            (uint16_t)(s.tap_row & 15));
          } else if (P.mode == kTc4Taps) {
            for (int k = 0; k < 3; ++k)
              ptx::tma_load_im2col_4d<PAIR>(dst + k * 128 * 128, &map_x, bar, ch, w0 * st - L.pad, h0 * st - L.pad, n0,
                                            (uint16_t)k, (uint16_t)(s.tap_row & 15));
          } else {
            for (int k = 0; k < tiles; ++k)
              ptx::tma_load_im2col_4d<PAIR>(dst + k * 128 * 128, &map_x, bar, ch + k * (I8 ? 128 : 64), w0 * st, h0 * st, n0, 0, 0);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 2) {
    // ============================================================ weight producer
    const int row0 = tile_n * (NT / 32) + (PAIR ? part * (NT / 64) : 0);   // blocks of 32 channels
    if (PAIR && P.packed) {
      if (jobs > 0 && ptx::elect_one()) {
        const int total = P.tiles_base + (BASE ? 0 : P.tiles_cond);
        for (int t = 0; t < total; t += 3) {
          const int tiles = min(3, total - t);
          const uint32_t bar = leader(&sh->b_full[t / 3]);
          expect(&sh->b_full[t / 3], (uint32_t)tiles * kTile);
          for (int k = t; k < t + tiles; ++k) {
            const bool cond = k >= P.tiles_base;
            const int tile = cond ? k - P.tiles_base : k;
            ptx::tma_load_5d<PAIR>(s_b + (size_t)k * kTile, cond ? &map_wc : &map_wb, bar,
                                   tile * (I8 ? 128 : 64), 0, 0, 0, row0);
          }
        }
      }
    } else if (ptx::elect_one()) {
      Cursor c{0, 0};
      bool ok = true, seen = false;
      const int rounds = P.resident ? (jobs > 0 ? 1 : 0) : jobs;
      for (int j = 0; j < rounds && ok; ++j) {
        Tc4Row next = row_at(table, lo);
        for (int i = lo; i < hi; ++i) {
          const Tc4Row s = next;
          if (i + 1 < hi) next = row_at(table, i + 1);
          if (!(s.flags & kRowBNew)) continue;
          if (!seen) ok = wait4_one(sh, prm.counters, &sh->b_empty[c.slot], c.par ^ 1u, 2);
          if (!ok) break;
          uint8_t* dst = s_b + (size_t)c.slot * P.stage_bytes;
          uint64_t* full = &sh->b_full[c.slot];
          c.next(P.nb);
          seen = ptx::mbar_test_wait(&sh->b_empty[c.slot], c.par ^ 1u);
          const int tiles = s.tap_row >> 4, bx = (int)s.bx, bstep = (int)s.bstep;
          const uint32_t bar = leader(full);
          const bool half = HALF && j == P.half_job && !P.resident;
          const CUtensorMap* map = (s.flags & kRowCond) ? &map_wc : &map_wb;
          if constexpr (HALF) map = half ? ((s.flags & kRowCond) ? &maps.half_wc : &maps.half_wb) : map;
          const int rows = row0 + (half ? group & 1 : 0);
          expect(full, (uint32_t)tiles * (half ? kTile / 2u : kTile));
          ptx::tma_load_5d<PAIR>(dst, map, bar, bx, 0, 0, 0, rows);
          if (tiles > 1) ptx::tma_load_5d<PAIR>(dst + kTile, map, bar, bx + bstep, 0, 0, 0, rows);
          if (tiles > 2) ptx::tma_load_5d<PAIR>(dst + 2 * kTile, map, bar, bx + 2 * bstep, 0, 0, 0, rows);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ============================================================ MMA issuer
    // (One lane picked by elect.sync runs the loop: an MMA then takes under 40 cycles to issue, against 50
    // predicated or in a branch on the lane.  A pair's MMAs are issued by its first CTA.)
    const uint32_t a0 = (ptx::smem_u32(s_a) >> 4) | 0x10000u, b0 = (ptx::smem_u32(s_b) >> 4) | 0x10000u;
    if constexpr (PAIR) {
      if (part == 0 && ptx::elect_one()) {
        const int kp = L.c_p % (I8 ? 128 : 64) == 0 ? 4 : L.c_p / (I8 ? 32 : 16);
        if (P.mode == kTc4Window) {
          if (P.packed && NT == 128) {
            if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Window, 2, 2>(prm, sh, a0, b0, tmem, group, jobs);
            else issue_jobs<NT, I8, BASE, HALF, kTc4Window, 1, 2>(prm, sh, a0, b0, tmem, group, jobs);
          } else if (kp == 4) issue_jobs<NT, I8, BASE, HALF, kTc4Window, 4>(prm, sh, a0, b0, tmem, group, jobs);
          else if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Window, 2>(prm, sh, a0, b0, tmem, group, jobs);
          else issue_jobs<NT, I8, BASE, HALF, kTc4Window, 1>(prm, sh, a0, b0, tmem, group, jobs);
        } else if (P.mode == kTc4Lattice) {
          if (kp == 4) issue_jobs<NT, I8, BASE, HALF, kTc4Lattice, 4>(prm, sh, a0, b0, tmem, group, jobs);
          else if (L.c_in == (I8 ? 256 : 128)) {
            if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Lattice, 2, 2>(prm, sh, a0, b0, tmem, group, jobs);
            else issue_jobs<NT, I8, BASE, HALF, kTc4Lattice, 1, 2>(prm, sh, a0, b0, tmem, group, jobs);
          } else {
            if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Lattice, 2, 1>(prm, sh, a0, b0, tmem, group, jobs);
            else issue_jobs<NT, I8, BASE, HALF, kTc4Lattice, 1, 1>(prm, sh, a0, b0, tmem, group, jobs);
          }
        } else if (P.mode == kTc4Rows2) {
          if (kp == 4) issue_jobs<NT, I8, BASE, HALF, kTc4Rows2, 4>(prm, sh, a0, b0, tmem, group, jobs);
          else if (L.c_in == (I8 ? 256 : 128)) {
            if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Rows2, 2, 2>(prm, sh, a0, b0, tmem, group, jobs);
            else issue_jobs<NT, I8, BASE, HALF, kTc4Rows2, 1, 2>(prm, sh, a0, b0, tmem, group, jobs);
          } else {
            if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Rows2, 2, 1>(prm, sh, a0, b0, tmem, group, jobs);
            else issue_jobs<NT, I8, BASE, HALF, kTc4Rows2, 1, 1>(prm, sh, a0, b0, tmem, group, jobs);
          }
        } else if (P.mode == kTc4Taps) {
          if (kp == 4) issue_jobs<NT, I8, BASE, HALF, kTc4Taps, 4>(prm, sh, a0, b0, tmem, group, jobs);
          else if (kp == 2) issue_jobs<NT, I8, BASE, HALF, kTc4Taps, 2>(prm, sh, a0, b0, tmem, group, jobs);
          else issue_jobs<NT, I8, BASE, HALF, kTc4Taps, 1>(prm, sh, a0, b0, tmem, group, jobs);
        } else if (!BASE) {
          issue_jobs<NT, I8, BASE, HALF, kTc4Chunks, 4>(prm, sh, a0, b0, tmem, group, jobs);
        }
      }
    } else if (jobs > 0 && ptx::elect_one()) {
      // a CTA of a cluster: its rows of the table
      const uint32_t idesc = I8 ? ptx::idesc_s8(128, NT) : ptx::idesc_bf16(128, NT);
      const uint32_t hi_w = (uint32_t)(ptx::smem_desc(0, 1024, 2) >> 32);
      const uint32_t a_size = (uint32_t)P.slot_bytes >> 4, b_size = (uint32_t)P.stage_bytes >> 4, a_step = (uint32_t)P.a_step, row_lo = (uint32_t)P.wp * 8u;
      bool ok = true;
      Cursor ca{0, 0}, cb{0, 0};
      int sa = 0, sb_base = 0, sb_cond = 0;                    // slots in use
      bool a_seen = false, b_seen = false;                     // the next row's slots were full when last looked at
      Tc4Row next = row_at(table, lo);
      for (int i = lo; i < hi; ++i) {
        const Tc4Row s = next;
        if (i + 1 < hi) next = row_at(table, i + 1);
        if (s.flags & kRowANew) {
          if (!a_seen) ok = wait4_one(sh, prm.counters, &sh->a_full[ca.slot], ca.par, 4);
          sa = ca.slot; ca.next(P.na);
        }
        if (s.flags & kRowBNew) {
          if (!b_seen) ok = ok && wait4_one(sh, prm.counters, &sh->b_full[cb.slot], cb.par, 5);
          if (s.flags & kRowCond) sb_cond = cb.slot; else sb_base = cb.slot;
          cb.next(P.nb);
        }
        if (!ok) break;
        if (i + 1 < hi) {
          // a look at the next row's barriers, whose answer arrives while this row's MMAs are issued
          a_seen = (next.flags & kRowANew) && ptx::mbar_test_wait(&sh->a_full[ca.slot], ca.par);
          b_seen = (next.flags & kRowBNew) && ptx::mbar_test_wait(&sh->b_full[cb.slot], cb.par);
        }
        const int sb = (s.flags & kRowCond) ? sb_cond : sb_base;
        const uint32_t a = a0 + (uint32_t)sa * a_size + s.a_off, b = b0 + (uint32_t)sb * b_size;
        const uint32_t d = tmem + ((s.flags & kRowR) ? (uint32_t)NT : 0u), acc = (s.flags & kRowInit) ? 0u : 1u;
        const int tiles = ((s.kind >> 4) & 3) + 1, nks = (s.kind & 3) + 1;
        const uint32_t b1 = b + s.b_off[0], b2 = b + s.b_off[1], b3 = b + s.b_off[2];
        if (s.kind & kKindTaps) {
          if (nks == 1) issue_taps<PAIR, I8, 0, 9, 0, 0, 1, 4, 0>(d, hi_w, a, row_lo, 8u, b, kTile >> 4, idesc, acc);
          else issue_taps<PAIR, I8, 0, 6, 0, 0, 2, 2, 0>(d, hi_w, a, row_lo, 8u, b, kTile >> 4, idesc, acc);
        } else if (nks == 4) issue_row<PAIR, I8, 4>(tiles, d, hi_w, a, a_step, b1, b2, b3, idesc, acc);
        else if (nks == 3) issue_row<PAIR, I8, 3>(tiles, d, hi_w, a, a_step, b1, b2, b3, idesc, acc);
        else if (nks == 2) issue_row<PAIR, I8, 2>(tiles, d, hi_w, a, a_step, b1, b2, b3, idesc, acc);
        else issue_row<PAIR, I8, 1>(tiles, d, hi_w, a, a_step, b1, b2, b3, idesc, acc);
        if (s.flags & kRowBFree) ptx::umma_commit(&sh->b_empty[sb]);
        if (s.flags & kRowAFree) ptx::umma_commit(&sh->a_empty[sa]);
      }
      if (ok) ptx::umma_commit(&sh->acc_full[0]);
    }
    __syncwarp();
  } else if (warp >= kEpiWarp0) {
    // ============================================================ epilogue
    const int et = (int)threadIdx.x - kEpiWarp0 * 32;
    for (int c = et; c < NT; c += kEpiThreads) {
      const int ch = tile_n * NT + c;
      if (ch < L.c_out) {
        if (I8) {
          s_q[c] = make_int4(prm.bn.q_gate_thr[ch], prm.bn.q_mul_base[ch], prm.bn.q_mul_full[ch], 0);
          s_o[c] = make_longlong2(add_half(prm.bn.q_off_base[ch], L.shift), add_half(prm.bn.q_off_full[ch], L.shift));
        } else {
          const ChannelConsts k = fold_channel(prm.bn, prm.delta, L.eps, ch);
          s_t[c] = k.t; s_t2[c] = k.t2; s_k[c] = make_float4(k.a1, k.b1, k.a2, k.b2);
        }
      }
    }
    ptx::named_bar_sync(2, kEpiThreads);
    const bool two_sided = !I8 && prm.bn.delta_high != nullptr;
    const int lo_q = L.relu ? 0 : -128;
    // 32 channels of a lane quadrant per warp: the 16 warps take a 128-channel job together; for 64 channels,
    // eight take the even jobs and eight the odd ones
    const int quad = warp & 3, eg = (warp - kEpiWarp0) >> 2;
    const int c0 = (NT == 128 ? eg : eg & 1) * 32;
    const int row = quad * 32 + lane;
    const uint32_t t_lane = tmem + ((uint32_t)(quad * 32) << 16);
    uint32_t active = 0, rows_active = 0;
    bool ok = true;
    if (!SPLIT) {
      // A thread holds, of every 16-row piece, two rows and the same eight channels (the weight tiles' row
      // order makes them consecutive): their constants stay in registers.
      const int ch = tile_n * NT + c0;
      const int q8 = (lane & 3) * 8, r4 = lane >> 2;
      float t[8];
      uint64_t a1[4], b1[4], a2[4], b2[4];                     // pairs of channels
      int qt[8], qm1[8], qm2[8];
      long long qo1[8], qo2[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int c = c0 + q8 + e;
        if (I8) {
          const int4 k = s_q[c];
          const longlong2 o = s_o[c];
          qt[e] = k.x; qm1[e] = k.y; qm2[e] = k.z; qo1[e] = o.x; qo2[e] = o.y;
        } else {
          t[e] = s_t[c];
          if (e & 1) {
            const float4 k = s_k[c - 1], l = s_k[c];
            a1[e / 2] = ptx::pack_f32x2(k.x, l.x); b1[e / 2] = ptx::pack_f32x2(k.y, l.y);
            a2[e / 2] = ptx::pack_f32x2(k.z, l.z); b2[e / 2] = ptx::pack_f32x2(k.w, l.w);
          }
        }
      }
      const uint32_t sel1 = lane & 1 ? 0x3715u : 0x6240u, sel2 = lane & 2 ? 0x3276u : 0x5410u;
      const bool has_res = !I8 && prm.residual != nullptr;
      for (int j = NT == 128 ? 0 : eg >> 1; j < jobs && ok; j += NT == 128 ? 1 : 2) {
        const int stage = j % kAcc;
        // (a half job's columns are the even or the odd blocks of 32 channels: warps of the others only wait)
        const bool half = HALF && j == P.half_job, mine = !half || (eg & 1) == (group & 1);
        const uint32_t t_col = t_lane + (uint32_t)(stage * 2 * NT + (half ? (eg >> 1) * 32 : c0));
        const uint32_t pos = (uint32_t)(job_pos(j) + row);
        const uint32_t n0 = P.div_ip.div(pos), rem = pos - n0 * (uint32_t)(P.wp * P.hp);
        const uint32_t h0 = P.div_wp.div(rem), w0 = rem - h0 * (uint32_t)P.wp;
        // pixel of this lane's row, or -1 (a padding position); the rows of the pieces take it from there
        const int own = (int)n0 < L.n && (int)h0 < L.ho && (int)w0 < L.wo ? (int)((n0 * L.ho + h0) * L.wo + w0) : -1;
        // (the residual comes to L2 while the sums are waited for)
        if (has_res && own >= 0 && ch < L.c_out) ptx::prefetch_l2(prm.residual + (long long)own * L.c_out + ch);
        ok = wait4(sh, prm.counters, &sh->acc_full[stage], (j / kAcc) & 1, 6);
        if (!ok) break;
        ptx::tc_fence_after();
        // (one instruction stream per kind of layer: every branch taken per element would cost as much as the
        // element's arithmetic)
        auto finish = [&](auto two_tag, auto res_tag) {
          [[maybe_unused]] constexpr bool kTwo = decltype(two_tag)::value;
          constexpr bool kRes = decltype(res_tag)::value;
          uint32_t bits = 0;                                   // byte i: the decisions of row r4 + 8i
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            int m[2];
            uint4 res[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              m[h] = __shfl_sync(0xffffffffu, own, r4 + 16 * i + 8 * h);
              if (kRes) {
                res[h] = make_uint4(0u, 0u, 0u, 0u);
                if (has_res && m[h] >= 0) res[h] = ptx::ld_global_16(prm.residual + (long long)m[h] * L.c_out + ch + q8);
              }
            }
            uint32_t out[2][4];
#pragma unroll
            for (int g = 0; g < 2; ++g) {                      // 16 columns at a time (registers)
              uint32_t p[8], r[8];
              const uint32_t t_p = t_col + ((uint32_t)(16 * i) << 16) + (uint32_t)(16 * g);
              __syncwarp();                                    // (the loads are .aligned; what is before them diverges)
              ptx::tmem_ld_frag16(t_p, p);
              if (has_cond) {
                ptx::tmem_ld_frag16(t_p + NT, r);
                ptx::tmem_ld_wait16(p, r);
              } else {
                ptx::tmem_ld_wait8(p);
#pragma unroll
                for (int e = 0; e < 8; ++e) r[e] = 0u;
              }
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                if constexpr (I8) {
                  int q[4];
#pragma unroll
                  for (int e = 0; e < 4; ++e) {
                    const int v = 4 * (e >> 1) + 2 * h + (e & 1), k = 4 * g + e;
                    const bool d = (int)p[v] >= qt[k];
                    if (d) bits |= 1u << (k + 8 * (2 * i + h));
                    q[e] = requantise(d ? qm2[k] : qm1[k], d ? qo2[k] : qo1[k], (int)p[v] + (d ? (int)r[v] : 0), L.shift);
                  }
                  out[h][g] = pack_s8(q, lo_q);
                } else {
#pragma unroll
                  for (int w = 0; w < 2; ++w) {
                    const int v = 4 * w + 2 * h, o = 2 * g + w, k = 2 * o;
                    const float p0 = __uint_as_float(p[v]), p1 = __uint_as_float(p[v + 1]);
                    // Eq. 1 under the batch norm of its path (Section 4), one fused multiply-add each, two
                    // channels per instruction
                    const uint64_t pp = ptx::pack_f32x2(p0, p1);
                    const uint64_t sum = ptx::add_f32x2(pp, ptx::pack_f32x2(__uint_as_float(r[v]), __uint_as_float(r[v + 1])));
                    float f0, f1, c0_, c1_;
                    ptx::unpack_f32x2(ptx::fma_f32x2(a2[o], sum, b2[o]), f0, f1);
                    ptx::unpack_f32x2(ptx::fma_f32x2(a1[o], pp, b1[o]), c0_, c1_);
                    // d = (P >= t) (and P <= t2); a NaN sum does not fire
                    bool d0 = p0 >= t[k], d1 = p1 >= t[k + 1];
                    if (kTwo) {
                      d0 = d0 && p0 <= s_t2[c0 + q8 + k];
                      d1 = d1 && p1 <= s_t2[c0 + q8 + k + 1];
                    }
                    if (d0) bits |= 1u << (k + 8 * (2 * i + h));
                    if (d1) bits |= 2u << (k + 8 * (2 * i + h));
                    float y0 = d0 ? f0 : c0_, y1 = d1 ? f1 : c1_;
                    if (kRes) {
                      const uint32_t x = o == 0 ? res[h].x : o == 1 ? res[h].y : o == 2 ? res[h].z : res[h].w;
                      y0 += __uint_as_float(x << 16); y1 += __uint_as_float(x & 0xffff0000u);
                    }
                    out[h][o] = pack_bf16(y0, y1);
                    if (L.relu) out[h][o] = relu_bf16x2(out[h][o]);
                  }
                }
              }
            }
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const long long at = (long long)m[h] * L.c_out + ch + q8;
              if (m[h] < 0) bits &= ~(255u << (8 * (2 * i + h)));
              else if constexpr (I8) *(uint2*)((uint8_t*)prm.y + at) = make_uint2(out[h][0], out[h][1]);
              else *(uint4*)((__nv_bfloat16*)prm.y + at) = make_uint4(out[h][0], out[h][1], out[h][2], out[h][3]);
            }
          }
          __syncwarp();
          // the four lanes of a row group exchange bytes: lane q gets the mask word of row r4 + 8q
          bits = __byte_perm(bits, __shfl_xor_sync(0xffffffffu, bits, 1), sel1);
          bits = __byte_perm(bits, __shfl_xor_sync(0xffffffffu, bits, 2), sel2);
          active += (uint32_t)__popc(bits);
          rows_active += bits != 0u ? 1u : 0u;
          const int m_word = __shfl_sync(0xffffffffu, own, r4 + q8);
          if (prm.mask && m_word >= 0) prm.mask[(long long)m_word * L.words + (ch >> 5)] = bits;
          return bits;
        };
        if (ch < L.c_out && mine) {                            // (uniform over the warp)
          if constexpr (BASE && !I8) {
            const uint32_t fired = finish(std::true_type{}, std::true_type{});
            if (__any_sync(0xffffffffu, fired != 0u))
              infinite_sums(prm, t_col, s_t + c0, s_t2 + c0, s_k + c0, ch, own);
          } else if (I8) finish(std::false_type{}, std::false_type{});
          else if (two_sided) finish(std::true_type{}, std::true_type{});
          else if (has_res) finish(std::false_type{}, std::true_type{});
          else finish(std::false_type{}, std::false_type{});
        }
        // the sums have been read: the accumulators go back to the issuers
        ptx::tc_fence_before();
        __syncwarp();
        // (not behind the last jobs: nobody waits for them, and the block may be gone)
        if (lane == 0 && j + kAcc < jobs) ptx::mbar_arrive_cluster_relaxed(leader(&sh->acc_empty[stage]));
      }
    }
    if constexpr (SPLIT) {
      // rows [part * rows, (part + 1) * rows) of the job are this CTA's to finish: four channels per thread
      constexpr int kLanes = NT / 4;                           // threads per row
      const int rows = split_rows(P, group);
      const uint32_t block = (uint32_t)rows * kSumPitch;       // a CTA's sums of those rows, of one path
      struct Item { long long at; int m; uint2 res; bool valid; };
      auto item = [&](int u) {
        Item t;
        const int lr = u / kLanes, cc = (u % kLanes) * 4;
        const uint32_t pos = (uint32_t)(group * 128 + part * rows + lr);
        const uint32_t n0 = P.div_ip.div(pos), rem = pos - n0 * (uint32_t)(P.wp * P.hp);
        const uint32_t h0 = P.div_wp.div(rem), w0 = rem - h0 * (uint32_t)P.wp;
        const int ch = tile_n * NT + cc;
        t.valid = u < rows * kLanes && jobs > 0 && (int)n0 < L.n && (int)h0 < L.ho && (int)w0 < L.wo && ch < L.c_out;
        t.m = t.valid ? (int)((n0 * L.ho + h0) * L.wo + w0) : 0;
        t.at = (long long)t.m * L.c_out + ch;
        t.res = make_uint2(0u, 0u);
        if (!I8 && prm.residual && t.valid) t.res = ptx::ld_global_8(prm.residual + t.at);
        return t;
      };
      Item next = item(et);                                    // (a residual is on its way while the sums are waited for)
      // This CTA's share of the sums goes to shared memory (the rings are idle once every MMA is done) ...
      ok = wait4(sh, prm.counters, &sh->acc_full[0], 0, 7);
      if (ok) {
        ptx::tc_fence_after();
        const int path = eg >> 1;                              // eight warps write P, eight R
        if (((path ? P.r_mask : P.p_mask) >> part) & 1) {
          uint32_t v[32];
          ptx::tmem_ld_nowait<32>(t_lane + (uint32_t)(path * NT + c0), v);
          ptx::tmem_ld_wait<32>(v);
          // (columns 2i, 2i+1 are channels 8*(i%4) + 2*(i/4), + 1 of the block: the weight tiles' row order)
          uint2* dst = (uint2*)(smem + kOffStages + ((unsigned)path * 128u + (unsigned)row) * kSumPitch + (unsigned)c0 * 4u);
#pragma unroll
          for (int i = 0; i < 16; ++i) dst[(i & 3) * 4 + (i >> 2)] = make_uint2(v[2 * i], v[2 * i + 1]);
        }
        ptx::tc_fence_before();
        ptx::fence_proxy_async();
      }
      // ... and from there, one copy per path, to the CTAs that finish its rows.  (Read by them through distributed shared
      // memory, 16 bytes a thread, they took 3,500 of a layer's 10,000 cycles, in flight together or not.)
      ok = !ptx::named_bar_or(3, kEpiThreads, !ok);
      if (P.sums_late) ptx::cluster_sync();                    // (their room is part of the rings: no MMA reads those any more)
      const int turn = warp - kEpiWarp0 + 1;                   // (one destination a warp, another one first in every CTA: all
      if (ok && turn <= P.split && lane < 2) {                 // sending to the first and then to the second took three times as long)
        const int to = (part + turn) & (P.split - 1), mine = lane ? P.r_mask : P.p_mask, others = ~(1 << to);
        if (to != part && ((mine >> part) & 1)) {
          const int slot = (lane ? __popc(P.p_mask & others) : 0) + __popc(mine & others & ((1 << part) - 1));
          ptx::bulk_copy_cluster(ptx::map_cluster(ptx::smem_u32(smem) + P.off_sums + (uint32_t)slot * block, (uint32_t)to),
                                 ptx::smem_u32(smem) + kOffStages + (uint32_t)lane * 128u * kSumPitch + (uint32_t)to * block, block,
                                 ptx::map_cluster(ptx::smem_u32(&sh->sums), (uint32_t)to));
        }
      }
      __syncwarp();
      ok = ok && wait4(sh, prm.counters, &sh->sums, 0, 9);
      for (int u = et; ok && u < rows * kLanes; u += kEpiThreads) {
        const Item t = next;
        const int lr = u / kLanes, cc = (u % kLanes) * 4, ch = tile_n * NT + cc;
        uint32_t w = 0;
        float pf[4] = {0.f, 0.f, 0.f, 0.f}, rf[4] = {0.f, 0.f, 0.f, 0.f};
        int pi[4] = {0, 0, 0, 0}, ri[4] = {0, 0, 0, 0};
        // the partial sums of the CTAs in order; this CTA's own are where it left them
        const uint32_t base = ptx::smem_u32(smem), in_row = (uint32_t)lr * kSumPitch + (uint32_t)cc * 4u;
        uint32_t from = base + P.off_sums + in_row, own = base + kOffStages + (uint32_t)part * block + in_row;
#pragma unroll
        for (int path = 0; path < 2; ++path, own += 128u * kSumPitch) {
          const int mask = path ? P.r_mask : P.p_mask;
          for (int peer = 0; peer < P.split; ++peer) {
            if (!((mask >> peer) & 1)) continue;
            const uint4 v = ptx::ld_shared_16(peer == part ? own : from);
            if (peer != part) from += block;
            if (path == 0) {
              if (I8) { pi[0] += (int)v.x; pi[1] += (int)v.y; pi[2] += (int)v.z; pi[3] += (int)v.w; }
              else { pf[0] += __uint_as_float(v.x); pf[1] += __uint_as_float(v.y); pf[2] += __uint_as_float(v.z); pf[3] += __uint_as_float(v.w); }
            } else {
              if (I8) { ri[0] += (int)v.x; ri[1] += (int)v.y; ri[2] += (int)v.z; ri[3] += (int)v.w; }
              else { rf[0] += __uint_as_float(v.x); rf[1] += __uint_as_float(v.y); rf[2] += __uint_as_float(v.z); rf[3] += __uint_as_float(v.w); }
            }
          }
        }
        if (u + kEpiThreads < rows * kLanes) next = item(u + kEpiThreads);
        if (t.valid) {
          if (I8) {
            int q[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int4 k = s_q[cc + e];
              const bool d = pi[e] >= k.x;
              if (d) w |= 1u << e;
              const longlong2 o = s_o[cc + e];
              q[e] = requantise(d ? k.z : k.y, d ? o.y : o.x, pi[e] + (d ? ri[e] : 0), L.shift);
            }
            *(uint32_t*)((uint8_t*)prm.y + t.at) = pack_s8(q, lo_q);
          } else {
            float v[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const bool d = pf[e] >= s_t[cc + e] && (!two_sided || pf[e] <= s_t2[cc + e]);
              if (d) w |= 1u << e;
              const float4 k = s_k[cc + e];
              const float full = fmaf(k.z, pf[e] + rf[e], k.w), base = fmaf(k.x, pf[e], k.y);
              v[e] = d ? full : base;
            }
            if (prm.residual) {
              v[0] += __uint_as_float(t.res.x << 16); v[1] += __uint_as_float(t.res.x & 0xffff0000u);
              v[2] += __uint_as_float(t.res.y << 16); v[3] += __uint_as_float(t.res.y & 0xffff0000u);
            }
            uint2 o = make_uint2(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]));
            if (L.relu) o = make_uint2(relu_bf16x2(o.x), relu_bf16x2(o.y));
            *(uint2*)((__nv_bfloat16*)prm.y + t.at) = o;
          }
        }
        // eight neighbouring threads hold the 32 channels of a mask word
        w <<= 4 * (lane & 7);
        w |= __shfl_xor_sync(0xffffffffu, w, 1);
        w |= __shfl_xor_sync(0xffffffffu, w, 2);
        w |= __shfl_xor_sync(0xffffffffu, w, 4);
        if (t.valid && (lane & 7) == 0) {
          active += (uint32_t)__popc(w);
          rows_active += w != 0u ? 1u : 0u;
          if (prm.mask) prm.mask[(long long)t.m * L.words + (ch >> 5)] = w;
        }
      }
    }
    active = __reduce_add_sync(0xffffffffu, active);
    rows_active = __reduce_add_sync(0xffffffffu, rows_active);
    if (lane == 0) {
      // the last warp sends the block's counts on their way, ahead of the cluster's last barrier
      atomicAdd(&sh->active, active); atomicAdd(&sh->rows_active, rows_active);
      __threadfence_block();
      if (atomicAdd(&sh->epi_done, 1u) == (uint32_t)kEpiWarps - 1u && !*(volatile uint32_t*)&sh->abort_flag) {
        const uint32_t all = atomicAdd(&sh->active, 0u), all_rows = atomicAdd(&sh->rows_active, 0u);
        if (all) atomicAdd(&prm.counters[CNT_ACTIVE], (unsigned long long)all);
        if (all_rows) atomicAdd(&prm.counters[CNT_ROWS_ACTIVE], (unsigned long long)all_rows);
      }
    }
  }
}

template <int NT, bool I8, bool PAIR, bool HALF>
__global__ void __launch_bounds__(kT4Threads, 1)
tc4_gated_conv_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ WeightMaps<HALF> maps,
                      const __grid_constant__ Tc4Params prm) {
  extern __shared__ uint8_t smem_raw[];
  constexpr bool SPLIT = !PAIR;
  ptx::grid_launch_dependents();
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  const LayerDims& L = prm.L;
  const Tc4Plan& P = prm.P;
  Shared4* sh = (Shared4*)smem;
  constexpr uint32_t kCols = PAIR ? 512 : 2 * NT;              // TMEM columns
  constexpr int kAcc = (int)kCols / (2 * NT);                  // accumulator pairs in them

  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const unsigned members = PAIR ? 2u : (unsigned)P.split;      // CTAs of a cluster
  const int part = (int)(blockIdx.x % members);                // rank in the cluster
  const int block = (int)(blockIdx.x / members), blocks = (int)(gridDim.x / members);
  // jobs of this cluster: a fixed column tile, every `groups`-th pixel tile (split layers: one job)
  const int tile_n = block % P.tiles_n, group = block / P.tiles_n, groups = blocks / P.tiles_n;
  const int jobs = HALF ? P.half_job + (group < 2 * P.half_tiles ? 1 : 0)
                   : group < P.tiles_m ? (P.tiles_m - group + groups - 1) / groups : 0;
  const bool has_cond = L.c_r > 0;

  if (warp == 0) {
    // (one barrier of a kind per lane: fifty in a row by one thread are a third of the set-up)
    if (lane < P.na) { ptx::mbar_init(&sh->a_full[lane], 1); ptx::mbar_init(&sh->a_empty[lane], 1); }
    if (lane < P.nb) { ptx::mbar_init(&sh->b_full[lane], 1); ptx::mbar_init(&sh->b_empty[lane], 1); }
    if (lane < kAcc) {
      ptx::mbar_init(&sh->acc_full[lane], 1);
      ptx::mbar_init(&sh->acc_empty[lane], (PAIR ? 2 : 1) * NT / 8);   // warps per job, of both CTAs of a pair
    }
    if (SPLIT && lane == 0) {
      // what the cluster sends here: P and R of this CTA's rows from every CTA that has some
      ptx::mbar_init(&sh->sums, 1);
      const int others = ~(1 << part);
      ptx::mbar_expect_tx(&sh->sums, (uint32_t)((__popc(P.p_mask & others) + __popc(P.r_mask & others)) * split_rows(P, group)) * kSumPitch);
    }
    if (lane == 0) { sh->abort_flag = 0; sh->active = 0; sh->rows_active = 0; sh->epi_done = 0; }
    ptx::fence_mbar_init();
  }
  if (threadIdx.x == 32 * 2) { ptx::prefetch_tensormap(&map_x); ptx::prefetch_tensormap(&maps.wb); ptx::prefetch_tensormap(&maps.wc); }
  // (the row table moves to shared memory: an indexed read of a kernel parameter costs hundreds of cycles)
  for (int i = (int)threadIdx.x - kEpiWarp0 * 32; i >= 0 && i < P.rows; i += kT4Threads)
    ((uint4*)(smem + kOffRows))[i] = ((const uint4*)P.row)[i];
  if (PAIR && P.base_rows && warp == kEpiWarp0 + kEpiWarps - 1) {
    // a first look, which costs nothing here; an open gate stays open for this launch whatever is written meanwhile
    const bool shut = gates_shut<NT, I8>(prm, tile_n, lane);
    if (lane == 0) sh->maybe_shut = shut ? 1u : 0u;
  }
  __syncwarp();
  if (warp == 1) { if (PAIR) ptx::tmem_alloc_pair(&sh->tmem_base, kCols); else ptx::tmem_alloc(&sh->tmem_base, kCols); }
  ptx::tc_fence_before();
  ptx::cluster_sync();
  ptx::tc_fence_after();
  // everything above touched only this cluster's own state
  ptx::grid_dependency_wait();
  const uint32_t tmem = sh->tmem_base;
  bool shut = false;
  if constexpr (PAIR) {
    // both CTAs of a pair have to choose alike: only where both saw shut gates, each looks at what counts
    if (P.base_rows && sh->maybe_shut && ptx::ld_cluster_4(ptx::smem_u32(&sh->maybe_shut), (uint32_t)(part ^ 1)))
      shut = gates_shut<NT, I8>(prm, tile_n, lane);
  }
  if (shut) {
    if constexpr (PAIR) {
      // the base rows move together
      const int i = (int)threadIdx.x;
      if (i < P.rows && ((P.base_mask >> i) & 1ull))
        ((uint4*)(smem + kOffRows))[__popcll(P.base_mask & ((1ull << i) - 1ull))] = ((const uint4*)P.row)[i];
      __syncthreads();
      run_roles<NT, I8, PAIR, HALF, true>(map_x, maps, prm, smem, warp, lane, part, tile_n, group, groups, jobs, tmem);
    }
  } else {
    run_roles<NT, I8, PAIR, HALF, false>(map_x, maps, prm, smem, warp, lane, part, tile_n, group, groups, jobs, tmem);
  }
  __syncwarp();
  if (SPLIT && P.sums_late && warp < kEpiWarp0) ptx::cluster_sync();
  // ---------------------------------------------------------------- teardown
  if (*(volatile uint32_t*)&sh->abort_flag) {
    // a wait gave up somewhere: let copies and MMAs that are still in flight finish (they take
    // microseconds) before the CTA's shared memory and TMEM go back
    const long long t_drain = clock64();
    while (clock64() - t_drain < 4000000ll) {}
  }
  __syncwarp();
  ptx::tc_fence_before();
  // No CTA leaves while a peer may still use its shared memory or TMEM.  (Every CTA has waited on its barrier `sums` for all
  // that is sent to it before it arrives here, so what a CTA sends has left its shared memory once all have arrived; stores to
  // global memory need not be waited for.  Where a CTA gave up waiting, the copies have the drain time above.)
  ptx::cluster_sync_relaxed();
  ptx::tc_fence_after();
  if (threadIdx.x == 0 && !*(volatile uint32_t*)&sh->abort_flag) {
    if (shut && part == 0) {
      // the jobs without conditional rows are taken from the totals below (the two halves of a job as one)
      const int halves = HALF && jobs > P.half_job ? 1 : 0, tiles = jobs - (halves & group & 1);
      atomicAdd(&prm.counters[CNT_TILES_TOTAL], 0ull - (unsigned long long)tiles);
      atomicAdd(&prm.counters[CNT_EXEC_MACS], 0ull - (unsigned long long)(jobs * NT - halves * (NT / 2)) * 256ull * (unsigned long long)(L.kh * L.kw) * L.c_r);
    }
    if (blockIdx.x == 0) {
      const unsigned long long tiles = (unsigned long long)P.tiles_m * P.tiles_n;
      atomicAdd(&prm.counters[CNT_CALLS], 1ull);
      atomicAdd(&prm.counters[CNT_TILES_TOTAL], has_cond ? tiles : 0ull);
      atomicAdd(&prm.counters[CNT_ROWS_TOTAL], (unsigned long long)L.m * L.words);
      atomicAdd(&prm.counters[CNT_EXEC_MACS], tiles * (PAIR ? 256ull : 128ull) * NT * (unsigned long long)(L.kh * L.kw) * L.c_in);
    }
  }
  if (warp == 1) {
    __syncwarp();
    if (PAIR) ptx::tmem_dealloc_pair(tmem, kCols); else ptx::tmem_dealloc(tmem, kCols);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
typedef CUresult (*EncodeIm2colFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const int*, const int*, cuuint32_t, cuuint32_t, const cuuint32_t*,
                                   CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                   CUtensorMapFloatOOBfill);

void* driver_fn(const char* name) {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult qr;
  if (cudaGetDriverEntryPointByVersion(name, &p, 12000, cudaEnableDefault, &qr) != cudaSuccess || qr != cudaDriverEntryPointSuccess)
    return nullptr;
  return p;
}

bool encode_x(CUtensorMap* map, const void* base, const LayerDims& L, const Tc4Plan& P) {
  static const EncodeIm2colFn fn = (EncodeIm2colFn)driver_fn("cuTensorMapEncodeIm2col");
  if (!fn) return false;
  const cuuint64_t eb = P.i8 ? 1 : 2;
  const cuuint64_t dims[4] = {(cuuint64_t)L.c_in, (cuuint64_t)L.w, (cuuint64_t)L.h, (cuuint64_t)L.n};
  const cuuint64_t str[3] = {L.c_in * eb, (cuuint64_t)L.w * L.c_in * eb, (cuuint64_t)L.h * L.w * L.c_in * eb};
  const int lower[2] = {-L.pad, -L.pad};
  // window modes: the box ends at the image's last column and row (at stride 2 a position more than there are outputs); else at
  // the last filter position.  A patch per filter row at stride 2: the last column, and the last filter position of a column.
  const int last = L.pad - (L.kw - 1);
  const bool window = P.mode == kTc4Window || P.mode == kTc4Lattice;
  const int upper[2] = {window || P.mode == kTc4Rows2 ? 0 : last, window ? 0 : last};
  const cuuint32_t st = P.mode == kTc4Window ? 1u : (cuuint32_t)L.stride;
  const cuuint32_t es[4] = {1, st, st, 1};
  return fn(map, P.i8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims,
            str, lower, upper, (cuuint32_t)(128 / eb), (cuuint32_t)P.patch_rows, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Weight tiles [output channel][K], the channels of each block of 32 in the order 8*(i%4) + 2*(i/4), + 1 for
// i = 0..15: accumulator columns 8k + 2q and + 1 are then channels 8q + 2k and + 1, so that the eight columns
// a thread gets of a block in the accumulator-fragment layout are eight consecutive channels.
// `blocks` of 32 channels to a copy.
bool encode_w(CUtensorMap* map, const void* base, const Tc4Plan& P, int c_out, int k_total, int blocks) {
  static const EncodeTiledFn fn = (EncodeTiledFn)driver_fn("cuTensorMapEncodeTiled");
  if (!fn) return false;
  const cuuint64_t eb = P.i8 ? 1 : 2, pitch = (cuuint64_t)k_total * eb;
  const cuuint64_t dims[5] = {(cuuint64_t)k_total, 2, 4, 4, (cuuint64_t)c_out / 32};
  const cuuint64_t str[4] = {pitch, 8 * pitch, 2 * pitch, 32 * pitch};
  const cuuint32_t box[5] = {(cuuint32_t)(128 / eb), 2, 4, 4, (cuuint32_t)blocks};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  return fn(map, P.i8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims,
            str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct RawRow {
  Tc4Row r;
  int a_key, b_key;      // which patch slot and which weight stage (unique numbers)
};

// The K loop of a job: every chunk and filter row, base channels into P, the others into R.
int raw_rows(const LayerDims& L, const Tc4Plan& P, RawRow* out) {
  const int eb = P.i8 ? 1 : 2, ck = 128 / eb, slice = 32 / eb;   // channels per chunk and per K slice
  const int chunks = L.c_in / ck, tile = (P.pair ? P.nt / 2 : P.nt) * 8;   // weight tile, 16-byte units
  int n = 0;
  // `tiles` pixel operands of nks slices from slice ks0 on, against the stage of `stage_tiles` tiles
  auto add = [&](int q, int r, int tiles, int ks0, int nks, bool cond, int bx, int bstep, int stage_tiles, int b_key) {
    if (n >= kTc4MaxRows) { n = kTc4MaxRows + 1; return (RawRow*)nullptr; }
    RawRow& o = out[n++];
    std::memset(&o, 0, sizeof(o));
    o.r.a_off = (uint16_t)((P.mode == kTc4Window ? r * P.wp * 8 : 0) + ks0 * 2);
    for (int s = 0; s < 3; ++s) o.r.b_off[s] = (uint16_t)(s * tile);
    o.r.bx = (uint16_t)bx; o.r.bstep = (uint16_t)bstep;
    o.r.flags = cond ? (uint8_t)(kRowR | kRowCond) : 0;
    o.r.kind = (uint8_t)((nks - 1) | ks0 << 2 | (tiles - 1) << 4);
    o.r.chunk = (uint8_t)q;
    o.r.tap_row = (uint8_t)(r | stage_tiles << 4);
    o.a_key = P.mode == kTc4Taps || P.mode == kTc4Rows2 ? q * 16 + r : q;
    o.b_key = b_key;
    return &o;
  };
  if (P.mode == kTc4Chunks) {
    for (int q = 0; q < chunks && n <= kTc4MaxRows; q += 3) {
      const int tiles = chunks - q < 3 ? chunks - q : 3;
      add(q, 0, tiles, 0, 4, false, q * ck, ck, tiles, 1000 + q);
    }
    return n;
  }
  for (int q = 0; q < chunks && n <= kTc4MaxRows; ++q) {
    const int kp = L.c_p - q * ck >= ck ? 4 : (L.c_p - q * ck > 0 ? (L.c_p - q * ck) / slice : 0);   // base slices of the chunk
    for (int r = 0; r < 3 && n <= kTc4MaxRows; ++r) {
      if (kp == 4) {
        add(q, r, 3, 0, 4, false, 3 * r * L.c_p + q * ck, L.c_p, 3, 1000 + q * 16 + r);
      } else if (kp == 0) {
        add(q, r, 3, 0, 4, true, 3 * r * L.c_r + q * ck - L.c_p, L.c_r, 3, 1000 + q * 16 + r);
      } else {
        // c_p < one chunk: a base tile holds the slices of 4/kp taps; one stage of three tiles for all taps
        // (kp = 1), or one for the first six taps and one of two tiles for the others (kp = 2)
        const int tpt = 4 / kp, second = kp == 2 && r == 2 ? 1 : 0;
        // (window mode: one entry for the taps of the first stage, issue_taps)
        const bool taps_entry = P.mode == kTc4Window && r == 0, covered = P.mode == kTc4Window && r > 0 && !second;
        RawRow* o = covered ? nullptr : add(q, r, 3, 0, kp, false, second * 3 * ck, ck, second ? 2 : 3, second);
        if (o && taps_entry) o->r.kind |= kKindTaps;
        if (o && !taps_entry)
          for (int s = 0; s < 3; ++s) {
            const int t = 3 * r + s;
            o->r.b_off[s] = (uint16_t)((t / tpt - second * 3) * tile + (t % tpt) * kp * 2);
          }
        add(q, r, 3, kp, 4 - kp, true, 3 * r * L.c_r, L.c_r, 3, 1000 + q * 16 + r);
      }
    }
  }
  return n;
}

// Rows [lo, hi) as one CTA (or pair) runs them, with their ring and accumulator flags.
void flag_rows(RawRow* st, int lo, int hi, int* a_count, int* b_count) {
  *a_count = *b_count = 0;
  bool seen[2] = {false, false};
  for (int i = lo; i < hi; ++i) {
    Tc4Row& s = st[i].r;
    const int path = s.flags & kRowR ? 1 : 0;
    if (!seen[path]) { s.flags |= kRowInit; seen[path] = true; }
    if (i == lo || st[i - 1].a_key != st[i].a_key) { s.flags |= kRowANew; ++*a_count; }
    if (i + 1 == hi || st[i + 1].a_key != st[i].a_key) s.flags |= kRowAFree;
    bool first = true, last = true;
    for (int k = lo; k < hi; ++k) {
      if (st[k].b_key != st[i].b_key) continue;
      if (k < i) first = false;
      if (k > i) last = false;
    }
    if (first) { s.flags |= kRowBNew; ++*b_count; }
    if (last) s.flags |= kRowBFree;
  }
}

// The base rows of a pair's jobs, as the jobs of a column tile whose gates cannot fire run them.
void plan_base(const RawRow* raw, Tc4Plan* P) {
  for (int i = 0; i < P->rows; ++i) {
    if (raw[i].r.flags & kRowCond) continue;
    P->base_mask |= 1ull << i;
    ++P->base_rows;
  }
}

// Stride-2 layers of pairs: windows over the four lattices of odd and even rows and columns, of pitch w' + 1 and h' + 1 (an odd
// lattice starts in the padding; an even one ends there).  Tap by tap the pixels of a job were copied nine times: 128->256
// channels at 28x28, 650 KB a job and CTA, 9,000 cycles of copies for 4,600 of MMAs.  Four of its patches are in use at a time
// (one by one for int8 with two packed chunks) and two more on their way, or a patch per filter row serves, of two lattices of
// pitch w' + 1 and h': six copies a chunk for four.  us a
// patch per filter row / per lattice (per lattice and one by one): 256->512 at 14x14 b128 21.6 / 17.6 (17.6), b64 13.0 / 12.0 (11.7),
// 128->256 at 28x28 b64 with G = 2 12.7 / 12.4 (11.7), with G = 4 13.6 / no room (12.7), 64->128 at 56x56 b128 18.2 / 18.5 (17.0).
bool plan_stride2(const LayerDims& L, Tc4Plan* P) {
  const int eb = P->i8 ? 1 : 2, ck = 128 / eb, tile = L.c_out <= 64 || (P->i8 && L.c_in <= ck) ? 4096 : 8192;
  if (L.w % 2 || L.h % 2) return false;
  if ((long long)L.n * (L.wo + 1) * (L.ho + 1) > 0x7fffffffll - 65536) return false;
  // a base path of less than a chunk: with packed weights that stay in shared memory
  const bool packed = L.c_p % ck != 0;
  if (packed && L.c_in > 2 * ck) return false;
  const int weights = (packed ? (9 * L.c_p + ck - 1) / ck + (9 * L.c_r + ck - 1) / ck : 9) * tile;
  const int room = (int)(kSmemBytes - 1024 - kOffStages) - weights, rows = (128 + L.wo + 2 + 7) / 8 * 8, slot = (rows * 128 + 1023) / 1024 * 1024;
  if (rows <= 256 && room >= (P->i8 && packed && L.c_in == 2 * ck ? 3 : 6) * slot) {
    P->mode = kTc4Lattice;
    P->wp = L.wo + 1; P->hp = L.ho + 1;
    P->loads = 1; P->patch_rows = rows; P->slot_bytes = slot;
  } else {
    const int slot2 = 2 * kLatticeRows * 128;
    if (L.wo < 2 || room < 2 * slot2) return false;            // (one pixel a row: half of the positions would be padding)
    P->mode = kTc4Rows2;
    P->wp = L.wo + 1; P->hp = L.ho;
    P->loads = 2; P->patch_rows = kLatticeRows; P->slot_bytes = slot2;
  }
  P->a_step = 8;
  return true;
}

template <int NT, bool I8, bool PAIR, bool HALF = false>
const void* instance() { return (const void*)tc4_gated_conv_kernel<NT, I8, PAIR, HALF>; }

}  // namespace

bool tc4_plan(const LayerDims& L, int in_dtype, int cond_mode, int sms, Tc4Plan* plan) {
  std::memset(plan, 0, sizeof(*plan));
  Tc4Plan P;
  std::memset(&P, 0, sizeof(P));
  if (in_dtype != CG_BF16 && in_dtype != CG_I8) return false;
  P.i8 = in_dtype == CG_I8;
  P.half_job = kNoHalfJob;
  const int eb = P.i8 ? 1 : 2, ck = 128 / eb, slice = 32 / eb;
  if (cond_mode == CG_COND_SKIP_TILES || cond_mode == CG_COND_COMPACT) return false;   // R is computed everywhere
  if (L.channel_tau > 0.f || (L.grouping && L.groups > 1)) return false;
  // 3x3 with pad 1 and 1x1 without gating of its input, any stride up to 8
  const bool k3 = L.kh == 3 && L.kw == 3 && L.pad == 1 && L.stride <= 8;
  const bool k1 = L.kh == 1 && L.kw == 1 && L.pad == 0 && L.stride <= 8 && L.c_r == 0;
  if (!k3 && !k1) return false;
  if (L.c_in % ck != 0 || L.c_in / ck > 255 || L.c_out % 32 != 0) return false;
  // base channels: whole chunks, or one or two K slices (a weight tile then holds whole taps)
  if (L.c_p % ck != 0 && L.c_p != slice && L.c_p != 2 * slice) return false;
  if ((long long)L.kh * L.kw * L.c_in > 65535) return false;
  P.mode = k1 ? kTc4Chunks : kTc4Taps;
  P.loads = 1; P.patch_rows = 128; P.a_step = 1024; P.slot_bytes = 3 * 128 * 128;
  P.wp = L.wo; P.hp = L.ho;
  if (k3 && L.stride == 1) {
    // a window: 128 positions and what the last tap reaches behind them, at most two loads of 256
    const int need = L.w <= 512 ? 128 + 2 * (L.w + 2) : 1 << 20;
    if (need <= 512) {
      P.mode = kTc4Window;
      P.wp = L.w + 1; P.hp = L.h + 1;
      P.loads = need <= 256 ? 1 : 2;
      P.patch_rows = ((need + P.loads - 1) / P.loads + 7) / 8 * 8;
      P.slot_bytes = (P.loads * P.patch_rows * 128 + 1023) / 1024 * 1024;
      P.a_step = 8;
    }
  }
  // (the extent of an image first: the products below stay within their types)
  const long long per_image = (long long)P.wp * P.hp;
  if (per_image > 0x3fffffffll || L.n * per_image > 0x7fffffffll - 65536) return false;
  const long long positions = L.n * per_image;
  P.div_ip.set((uint32_t)per_image); P.div_wp.set((uint32_t)P.wp);
  const int tiles128 = (int)((positions + 127) / 128);
  const int tn64 = (L.c_out + 63) / 64, tn128 = (L.c_out + 127) / 128;

  P.split = 1;
  int room = (int)(kSmemBytes - 1024 - kOffStages);
  RawRow raw[kTc4MaxRows];
  // (1x1 layers of up to three chunks have one row and nothing to share: as pairs they end without the exchange of
  // sums, 28x28 x 64 -> 128, one image, 8.5 and 5.0 us)
  const bool one_row = P.mode == kTc4Chunks && L.c_in <= 3 * ck;
  // Where a job's K loop is short, or only two CTAs could share it, pairs end sooner: they have no exchange of sums, but
  // their epilogue of 256 pixels waits longer for a residual.  us shared / as pairs (and with a residual), by MMAs a job:
  //   up to 36: 56x56 x 64 7.0 / 5.9, 28x28 x 64 6.3 / 6.0 (6.3 / 6.4), 56x56 x 64->128 stride 2 7.9 / 6.0, 14x14 x 256->512
  //     1x1 6.9 / 5.2; the pixels of a single job are shared sooner, 5x5 x 64 5.4 / 5.9 (5.2 / 6.1); with
  //     many columns, too: 128 x 512->1024, a classifier, is 5.6 as pairs in a chain of itself and 7.6 shared, but behind the
  //     other layers of a network 18.9 and 14.9 between events, a pass of one image 178.9 and 176.3;
  //   up to 72: 2 x 28x28 x 128 8.5 / 7.5, one image (14 jobs) 7.9 / 7.5 (7.9 / 8.1), 28x28 x 128->256 stride 2 8.1 / 6.5;
  //     eight CTAs to a job are faster, 3 x 14x14 x 128 (10 jobs) 6.9 / 7.4 (6.9 / 8.1);
  //   two CTAs: 8 x 14x14 x 256 10.7 / 8.5, 5 x 14x14 x 256 10.6 / 8.1 (10.6 / 8.7), 51 x 5x8 x 512->192 14.3 / 12.0;
  //   else shared: 14x14 x 256 7.5 / 8.1 (7.5 / 8.4), 7x7 x 512 7.3 / 11.5.
  const long long small = (long long)tiles128 * tn64, mmas = (long long)L.kh * L.kw * L.c_in / slice;
  const bool as_pairs = small * 4 > sms * 7 / 8 ||
                        (mmas <= 72 && tiles128 >= 2 && small >= (L.has_residual ? 16 : 14)) ||
                        (mmas <= 72 && !L.has_residual && (mmas <= 36 ? tiles128 >= 2 : L.stride == 2));
  if (!one_row && !as_pairs && small * 2 <= sms) {
    // Fewer jobs of 128 pixels and 64 channels than half the SMs: their K loops are shared, as far as all clusters
    // are on the chip at once.  Measured with 148 SMs: 32 clusters of 4 are, 15 of 8 are and 16 are not (9.2 against
    // 16.5 us for 4 x 7x7 x 512).  14 and 15 clusters of 8 gain nothing over 4 (4 x 7x7 x 512 -> 448 9.2 and 9.4 us, 6 x 7x7
    // x 512 -> 320 9.4 and 9.3), so the line of 8 lies at 13, clear of the edge.
    // Eight CTAs need sixteen rows, or exactly eight: with 9 or 12 the exchange costs what the shorter loops save (14x14 x
    // 256 7.5 us with 4 and 8; 28x28 x 128, 8 rows, 8.0 and 7.8; 9x9 x 128 7.0 and 6.5).
    P.nt = 64; P.tiles_m = tiles128; P.tiles_n = tn64;
    P.rows = raw_rows(L, P, raw);
    if (P.rows > kTc4MaxRows) return false;
    for (int s = 2; s <= kTc4MaxSplit; s *= 2)
      if (small * s <= (s == 8 ? sms * 3 / 4 : (s == 4 ? sms * 7 / 8 : sms)) &&
          (P.rows >= (s == 8 ? 16 : s) || P.rows == s))
        P.split = s;
    int total = 0, done = 0, s = 1;
    auto cost = [&](int i) {                                   // MMAs
      const int k = raw[i].r.kind, nks = (k & 3) + 1;
      return k & kKindTaps ? (nks == 1 ? 9 : 12) : nks * (((k >> 4) & 3) + 1);
    };
    for (int i = 0; i < P.rows; ++i) total += cost(i);
    for (int i = 0; i < P.rows; ++i) {
      if (s < P.split && i > P.lo[s - 1] && (done * P.split >= total * s || P.rows - i <= P.split - s)) P.lo[s++] = (uint16_t)i;
      done += cost(i);
    }
    P.lo[P.split] = (uint16_t)P.rows;
    P.grid = P.tiles_m * P.tiles_n * P.split;
  } else {
    // CTA pairs: each SM then fetches and holds half of the weights.  128 channels per job unless the layer
    // has fewer or the rounds of jobs come out shorter with 64: such a job takes about 0.85 of the time (512@4x4
    // b256: 3 rounds of 64 36.1 us, 2 rounds of 128 27.6; 128->256 stride 2: 19.0 and 15.7).  int8 layers of one chunk, whose epilogue is the longer
    // part: 64 (128@28x28 b64 15.6 and 15.8 us with 128, b20 9.7 and 10.0); with more chunks 128 is faster (256@14x14 b128
    // 20.4 and 19.3, 512@7x7 b128 21.1 and 18.8).
    P.pair = 1;
    const int pairs = sms / 2;
    int tiles256 = (int)((positions + 255) / 256);
    auto rounds = [&](int tn) { return tn > pairs ? 1e30 : (double)((tiles256 + pairs / tn - 1) / (pairs / tn)); };
    if (k3 && L.stride == 2 && plan_stride2(L, &P)) {
      // a third or two of the patch bytes, and more positions: not where that makes more than half as many rounds again
      const double taps = rounds(tn128);
      const long long padded = (long long)L.n * P.wp * P.hp;
      const int before = tiles256;
      tiles256 = (int)((padded + 255) / 256);
      if (rounds(tn128) > 1.5 * taps) {
        tiles256 = before;
        P.mode = kTc4Taps; P.wp = L.wo; P.hp = L.ho; P.loads = 1; P.patch_rows = 128; P.slot_bytes = 3 * 128 * 128; P.a_step = 1024;
      }
      P.div_ip.set((uint32_t)(P.wp * P.hp)); P.div_wp.set((uint32_t)P.wp);
    }
    P.nt = ((P.i8 && L.c_in <= ck) || L.c_out <= 64 || rounds(tn64) * 0.85 < rounds(tn128)) ? 64 : 128;
    P.tiles_m = tiles256; P.tiles_n = P.nt == 64 ? tn64 : tn128;
    if (P.tiles_n > pairs) return false;
    P.rows = raw_rows(L, P, raw);
    if (P.rows > kTc4MaxRows) return false;
    const int groups = pairs / P.tiles_n;
    // A last round that less than half of the pairs take part in: its jobs as two of 64 columns each, which take two thirds
    // of the time (43 cycles an MMA for 64).
    const int left = P.tiles_m % groups;
    if (P.nt == 128 && P.tiles_m > groups && left > 0 && 2 * left <= groups) { P.half_job = P.tiles_m / groups; P.half_tiles = left; }
    P.grid = (groups < P.tiles_m ? groups : P.tiles_m) * P.tiles_n * 2;
    P.lo[1] = (uint16_t)P.rows;
  }
  int max_a = 0, max_b = 0;
  for (int s = 0; s < P.split; ++s) {
    int a, b;
    flag_rows(raw, P.lo[s], P.lo[s + 1], &a, &b);
    if (a > max_a) max_a = a;
    if (b > max_b) max_b = b;
    for (int i = P.lo[s]; i < P.lo[s + 1]; ++i) {
      if (raw[i].r.flags & kRowR) P.r_mask |= (uint8_t)(1 << s);
      else P.p_mask |= (uint8_t)(1 << s);
    }
  }

  if (P.mode == kTc4Lattice) max_a = 4 * (L.c_in / ck);        // (not in the table)

  P.stage_bytes = 3 * (P.pair ? P.nt / 2 : P.nt) * 128;
  // a cluster's CTA: room for the sums that are sent to it, and for its own behind the rings' start
  const unsigned sums_bytes = P.pair ? 0u : (unsigned)(__builtin_popcount(P.p_mask) + __builtin_popcount(P.r_mask)) * (128u / (unsigned)P.split) * kSumPitch;
  // (within the rings' room, and one cluster barrier later, where the job's patches would not all fit beside it: tap by tap
  // 256->512 at 14x14, one image, 8.1 us beside the rings)
  const int slots_wanted = max_a < kMaxNA ? max_a : kMaxNA, stages_wanted = max_b < 3 ? max_b : 3;
  P.sums_late = !P.pair && P.mode == kTc4Taps && room - (int)sums_bytes < slots_wanted * P.slot_bytes + stages_wanted * P.stage_bytes;
  if (!P.sums_late) room -= (int)sums_bytes;

  // shared memory: resident weights if they leave room for three patch slots, else rings of both
  const int clusters = P.grid / (P.pair ? 2 : P.split);
  const int jobs = P.pair ? (P.tiles_m + clusters / P.tiles_n - 1) / (clusters / P.tiles_n) : 1;
  // 128 channels with a base path of less than a chunk, 128 to a job: whole tiles per tap and chunk are half empty and do not
  // fit, packed to 64 K elements each they do.  Streamed, they come to 240 KB a job and CTA, 83 bytes a cycle with what a
  // pair's MMAs fetch of each other's weights: 5,300 cycles a job, 4,600 of MMAs.
  const int tile_bytes = (P.pair ? P.nt / 2 : P.nt) * 128;
  const int tb = (9 * L.c_p + ck - 1) / ck, tc = (9 * L.c_r + ck - 1) / ck;
  if (P.mode == kTc4Lattice || P.mode == kTc4Rows2 ? L.c_p % ck != 0
                            : P.pair && P.mode == kTc4Window && P.nt == 128 && L.c_in == 2 * ck && L.c_p < ck && L.c_r > 0 &&
                                  room - (tb + tc) * tile_bytes >= 2 * P.slot_bytes) {
    P.packed = 1; P.resident = 1;
    P.tiles_base = tb; P.tiles_cond = tc;
    P.nb = (tb + tc + 2) / 3;
  } else if (max_b <= kMaxNB && jobs > 1 && room - max_b * P.stage_bytes >= (P.mode == kTc4Lattice ? 6 : P.mode == kTc4Rows2 ? 2 : 3) * P.slot_bytes) {
    P.resident = 1;
    P.nb = max_b;
  } else {
    // (three weight stages at least: a base stage stays while conditional ones pass)
    int na = P.mode == kTc4Lattice ? kLatticeSlots : P.mode == kTc4Window ? 3 : 2;
    if (na > max_a * jobs) na = max_a * jobs;
    while (na > (P.mode == kTc4Lattice ? 6 : 2) && room - na * P.slot_bytes < (P.mode == kTc4Lattice ? 3 : 4) * P.stage_bytes) --na;
    if (!P.pair && na > 1 && room - na * P.slot_bytes < 3 * P.stage_bytes) --na;
    P.nb = (room - na * P.slot_bytes) / P.stage_bytes;
    if (P.nb < 3) return false;
    if (P.nb > kMaxNB) P.nb = kMaxNB;
    if (P.nb > max_b * jobs) P.nb = max_b * jobs;
  }
  const int weights = P.packed ? (tb + tc) * tile_bytes : P.nb * P.stage_bytes;
  P.na = (room - weights) / P.slot_bytes;                      // what is left goes to patches
  if (P.na > kMaxNA) P.na = kMaxNA;
  if (P.na < 1 || (P.pair && P.na < 2 && max_a * jobs > 1)) return false;
  if (P.pair && L.c_r > 0 && cond_mode == CG_COND_AUTO) plan_base(raw, &P);
  for (int i = 0; i < P.rows; ++i) {
    P.row[i] = raw[i].r;
  }
  P.positions = (int)((long long)L.n * P.wp * P.hp);
  P.off_b = kOffStages;
  P.off_a = kOffStages + (unsigned)(P.packed ? weights : P.nb * P.stage_bytes);
  P.smem_bytes = kSmemBytes;
  if (!P.pair) P.off_sums = P.sums_late ? kOffStages + 2u * 128u * kSumPitch : kSmemBytes - 1024 - sums_bytes;
  P.valid = 1;
  *plan = P;
  return true;
}

int launch_tc4(const LayerDims& L, const Tc4Plan& P, Tc4Maps* maps, const void* x, const void* w_base,
               const void* w_cond, const cg_bn_params& bn, const float* delta, const void* residual, void* y,
               uint32_t* mask, unsigned long long* counters, cudaStream_t stream) {
  if (!P.valid) return (int)cudaErrorInvalidValue;
  Tc4MapSet* ms = nullptr;
  const Tc4MapSet* same_weights = nullptr;                     // (x alone is new: the weights' maps, up to four, are there)
  for (int i = 0; i < Tc4Maps::kEntries; ++i) {
    Tc4MapSet* c = &maps->set[i];
    if (!c->key[0] || c->key[1] != w_base || c->key[2] != w_cond) continue;
    same_weights = c;
    if (c->key[0] == x) { ms = c; break; }
  }
  if (!ms) {
    ms = &maps->set[maps->next];
    maps->next = (maps->next + 1) % Tc4Maps::kEntries;
    ms->key[0] = nullptr;
    if (!encode_x(&ms->x, x, L, P)) return (int)cudaErrorInvalidValue;
    if (same_weights) {
      ms->wb = same_weights->wb; ms->wc = same_weights->wc;
      ms->half_wb = same_weights->half_wb; ms->half_wc = same_weights->half_wc;
    } else {
      const int taps = L.kh * L.kw;
      const int blocks = P.pair ? P.nt / 64 : P.nt / 32;
      const bool halves = P.half_job < kNoHalfJob;
      if (!encode_w(&ms->wb, w_base, P, L.c_out, taps * L.c_p, blocks)) return (int)cudaErrorInvalidValue;
      ms->wc = ms->half_wb = ms->half_wc = ms->wb;
      if (L.c_r > 0 && !encode_w(&ms->wc, w_cond, P, L.c_out, taps * L.c_r, blocks)) return (int)cudaErrorInvalidValue;
      if (halves && !encode_w(&ms->half_wb, w_base, P, L.c_out, taps * L.c_p, blocks / 2)) return (int)cudaErrorInvalidValue;
      if (halves && L.c_r > 0 && !encode_w(&ms->half_wc, w_cond, P, L.c_out, taps * L.c_r, blocks / 2)) return (int)cudaErrorInvalidValue;
    }
    ms->key[0] = x; ms->key[1] = w_base; ms->key[2] = w_cond;
  }
  Tc4Params prm;
  prm.L = L; prm.P = P; prm.bn = bn; prm.delta = delta;
  prm.residual = static_cast<const __nv_bfloat16*>(residual);
  prm.y = y; prm.mask = mask; prm.counters = counters;
  prm.x = static_cast<const __nv_bfloat16*>(x); prm.w_cond = static_cast<const __nv_bfloat16*>(w_cond);
  const bool half = P.half_job < kNoHalfJob;             // (pairs of 128 columns)
  const int which = half ? (P.i8 ? 9 : 8) : (P.nt == 128 ? 1 : 0) | (P.i8 ? 2 : 0) | (P.pair ? 4 : 0);
  static const void* const kernels[10] = {
      instance<64, false, false>(), nullptr, instance<64, true, false>(), nullptr,
      instance<64, false, true>(), instance<128, false, true>(), instance<64, true, true>(), instance<128, true, true>(), instance<128, false, true, true>(), instance<128, true, true, true>()};
  const void* kernel = kernels[which];
  if (!kernel) return (int)cudaErrorInvalidValue;
  static bool attr_set[64][10] = {};   // (the attribute is per device and kernel instance)
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return (int)cudaErrorInvalidDevice;
  if (!attr_set[dev][which]) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
    if (e != cudaSuccess) return (int)e;
    attr_set[dev][which] = true;
  }
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3((unsigned)P.grid, 1, 1);
  cfg.blockDim = dim3((unsigned)kT4Threads, 1, 1);
  cfg.dynamicSmemBytes = P.smem_bytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = P.pair ? 2u : (unsigned)P.split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  WeightMaps<true> maps_half = {ms->wb, ms->wc, ms->half_wb, ms->half_wc};
  WeightMaps<false> maps_all = {ms->wb, ms->wc};
  void* args[3] = {&ms->x, half ? (void*)&maps_half : (void*)&maps_all, &prm};
  const cudaError_t e = cudaLaunchKernelExC(&cfg, kernel, args);
  if (e != cudaSuccess) return (int)e;
  return (int)cudaGetLastError();
}

}  // namespace cg
