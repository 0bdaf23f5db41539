// Window tensor-core path of the channel-gated layer (tc4_conv.cu): plan and launcher.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace cg {

constexpr int kTc4MaxRows = 64;
constexpr int kTc4MaxSplit = 8;

// One row of a job's K loop: up to three weight tiles (128 K-bytes of the CTA's output channels) times the
// matching pixel operands -- the three taps of a filter row on one input-channel chunk, or, for 1x1 layers,
// up to three chunks -- with 1 to 4 MMAs of 32 K-bytes each.
struct alignas(16) Tc4Row {
  uint16_t a_off;      // operand start within the patch slot, 16-byte units (the tiles follow a_step apart)
  uint16_t b_off[3];   // operand starts within the weight stage, 16-byte units
  uint16_t bx;         // K coordinate of the stage's first weight tile (elements)
  uint16_t bstep;      // K distance of its tiles
  uint8_t flags;       // kRow* bits
  uint8_t kind;        // MMAs per tile - 1 | first slice of the patch << 2 | tiles - 1 << 4 | kKindTaps
  uint8_t chunk;       // first input-channel chunk
  uint8_t tap_row;     // filter row | weight tiles of the stage << 4
};
static_assert(sizeof(Tc4Row) == 16, "row table");

enum : uint8_t {
  // (the producers read kRowANew, kRowBNew and kRowCond; the others are for the issuer of a cluster's CTA: a pair's has no table)
  kRowR = 1,        // accumulates into R (else P)
  kRowInit = 2,     // first row into its accumulator: overwrites it
  kRowANew = 4, kRowAFree = 8,     // takes the next patch slot / is the last to read its slot
  kRowBNew = 16, kRowBFree = 32,   // the same for the weight stage
  kKindTaps = 64,   // (in `kind`) the first taps of the base path of a window, several per weight tile
  kRowCond = 64     // the weights come from W_cond (else W_base)
};

enum { kTc4Window = 0, kTc4Taps = 1, kTc4Chunks = 2, kTc4Lattice = 3, kTc4Rows2 = 4 };
constexpr int kNoHalfJob = 1 << 30;

struct Tc4Plan {
  int valid;
  int i8;
  int pair;              // 1: CTA pairs (256 pixels per job); 0: `split` CTAs share the K loop of a 128-pixel job
  int nt;                // output channels per job: 64 or 128
  int mode;              // kTc4Window, kTc4Taps, kTc4Chunks, kTc4Lattice, kTc4Rows2: what a patch slot holds
  int wp, hp;            // pitch of the stacked pixel space: window mode w + pad, h + pad; stride-2 windows w' + 1 and h' + 1 or h'; else w', h'
  FastDiv div_ip, div_wp;   // by wp * hp and by wp
  int positions;         // n * wp * hp
  int patch_rows;        // pixels per patch load
  int slot_bytes;        // patch slot: one or two loads of a window, two of a filter row (kTc4Rows2), or up to three of 128 pixels
  int loads;             // window modes: loads per slot
  int a_step;            // distance of a row's pixel operands, 16-byte units
  int na, nb;            // ring depths: patch slots, weight stages
  int stage_bytes;       // weight stage of one CTA
  int resident;          // the weights of a column tile stay in shared memory
  int packed, tiles_base, tiles_cond;   // ... as tiles of consecutive K elements of W_base and of W_cond, three to a barrier
  int tiles_m, tiles_n;  // jobs
  int half_job, half_tiles;   // job of a pair that has half of the columns (kNoHalfJob: none), and how many jobs are halved
  int split;             // 1, 2, 4 or 8
  int grid;
  int rows;              // entries of row[] in use
  uint16_t lo[kTc4MaxSplit + 1];   // rows [lo[s], lo[s+1]) belong to CTA s of a cluster
  // jobs of a column tile whose gates cannot fire (pairs) run the base rows only
  int base_rows;                   // 0: all jobs run all rows
  unsigned long long base_mask;    // which rows
  uint8_t p_mask, r_mask;          // which CTAs of a cluster add to P / to R
  int sums_late;         // the sums that a cluster exchanges lie within the rings
  unsigned off_b, off_a, off_sums, smem_bytes;
  Tc4Row row[kTc4MaxRows];
};

struct Tc4MapSet {
  const void* key[3];    // x, w_base, w_cond the maps were encoded for
  CUtensorMap x, wb, wc, half_wb, half_wc;
};

struct Tc4Maps {
  static constexpr int kEntries = 8;
  Tc4MapSet set[kEntries];
  int next;
};

bool tc4_plan(const LayerDims& L, int in_dtype, int cond_mode, int sms, Tc4Plan* plan);
int launch_tc4(const LayerDims& L, const Tc4Plan& plan, Tc4Maps* maps, const void* x, const void* w_base,
               const void* w_cond, const cg_bn_params& bn, const float* delta, const void* residual, void* y,
               uint32_t* mask, unsigned long long* counters, cudaStream_t stream);

}  // namespace cg
