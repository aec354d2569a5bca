// Subsampled global attention (Sec. 4.3 of the AVGGT paper) as one fused,
// warp-specialised flash-style kernel for sm_100a; the same kernel runs frame
// attention (Sec. 4.2) as many small dense problems.
//
// A work item is two tiles of 128 query rows of one head.  One CTA per SM walks
// over the work items; the next item's loads and first product run under the
// current item's last step, and the epilogue of an item comes after the first
// step of the next one, when its last product has long completed.
// Roles (20 warps):
//   warps 0-15  softmax.  Warp 8 t + 4 h + q works on query tile t, rows
//               [32 q + 16 h, 32 q + 16 h + 16), all 112 columns of a key step.
//               It reads tensor memory in the 16-lane shapes, which spread a row
//               over the four threads of a quad (two rows per thread): a row's
//               maximum is two shuffles away and every row lives in one warp.  Four softmax warps per scheduler keep the exponential unit
//               busy while others wait on tensor memory or barriers.
//   warp  16    TMA producer: Q tiles once per work item (two places), then the compacted
//               K/V of the head through a ring of shared-memory stages (128-byte swizzle), then, for the
//               epilogue, the query rows' own K and V and the head's mean pair; it also writes the record of the item
//               (ItemInfo)
//   warps 17-18 MMA issuers, one per query tile: S_t = Q_t Kc_j^T and
//               O_t += P_t Vc_j with tcgen05.mma, bf16 operands, fp32
//               accumulators in tensor memory
//   warp  19    allocates tensor memory (and completes the fifth warpgroup so that registers can
//               be moved to the softmax warpgroups)
// Tensor memory per tile (256 columns): two places for S and P that alternate (see kColSOdd), O (64) and the row
// sums of P (16).  A softmax thread pulls its 56 scores of S into registers and the warp frees its rows at once,
// so the next Q K^T runs under the exponentials; P V of step j runs under the softmax of step j+1.  Two
// blocks of 8 key columns in fourteen take their exponentials from a polynomial on
// the FMA pipe.  The accumulator is rescaled lazily: only when the running
// maximum grew by more than 2^8 since the last rescale.  The epilogue folds the
// diagonal and the mean-fill column into the same normalisation:
//   O = (a_S O_S + p_d v_i + p_m vmean) / (a_S l_S + p_d + p_m).
#include <cmath>
#include <cstddef>
#include <mutex>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "tmap.h"

namespace avggt {

namespace {

constexpr int kTileQ = 128;      // query rows per tile
constexpr int kQTiles = 2;       // tiles per CTA
constexpr int kTileKV = 112;     // keys per step
constexpr int kBlocks = kTileKV / 8;   // blocks of 8 key columns in a step
constexpr int kHeadDim = 64;
constexpr uint32_t kTileBytes = kTileQ * kHeadDim * 2;      // 16 KiB: one tile of 128 query rows
constexpr uint32_t kKeyTileBytes = kTileKV * kHeadDim * 2;  // 14 KiB: one tile of keys or values, one ring stage
static_assert(kKeyTileBytes % 1024 == 0, "swizzle atoms");
constexpr uint32_t kOnesBytes = 2 * 1024;                   // the block of value columns 64..79 (ones_block)
// K ring and V ring depth.  2, 3, 4 and 5 stages measured the same (layer of 100 frames 22.44, 22.48, 22.47 and 22.47 ms, frame
// attention of 100 frames 1099, 1102, 1105 and 1107 us); three leave room for the query rows' own K and V.
#ifndef AVGGT_STAGES
#define AVGGT_STAGES 3
#endif
constexpr int kStages = AVGGT_STAGES;
constexpr int kThreads = 640;
constexpr int kSoftmaxWarps = 16;
constexpr int kTmaWarp = 16;
constexpr int kMmaWarp = 17;
constexpr int kTmemWarp = 19;
constexpr uint32_t kTmemCols = 512;
// Tensor memory of a query tile (256 columns): scores and probabilities of the even steps of the tile, S at 0 and P at 0
// (over the scores it was computed from); of the odd steps, S at 64 and P at 112; O at 176, the row sums of P at 240.
// P of a step and S of the next one never share a column, so a step's Q K^T needs only that the previous step's scores
// have been read.
constexpr uint32_t kTmemTileStride = 256;
constexpr uint32_t kColSOdd = 64, kColPOdd = 112, kColO = 176, kColL = kColO + kHeadDim;
constexpr int kPvCols = kHeadDim + 16;   // N of P V: the value columns and the block whose first column is all ones
static_assert(kTileKV <= kColPOdd && kTileKV / 2 <= kColSOdd && kColSOdd + kTileKV <= kColO && kColPOdd + kTileKV / 2 <= kColO &&
              kColO + kPvCols <= kTmemTileStride, "tensor memory of a tile");
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleThreshold = 8.0f;   // log2 units
// The tensor core truncates when it accumulates: a sum of many positive terms comes out short by up to 2^-24 for each of the
// seven products of a step (measured 1.8e-3 after 4,086 steps, as large as a bf16 rounding step).  Every so many steps the
// row sums are therefore moved to the next column, to which P V adds exact zeros; what is left of the error is 2.7e-5.  (O itself is
// accumulated the same way and comes out short by as much as that or more, so that the two partly cancel: against 64 bits the
// outputs are no further off than with the sums in 32-bit registers, dense layer of 100 frames 1.656e-3 against 1.658e-3.)
constexpr int kFlushSteps = 64;
static_assert(kFlushSteps > 1, "an item's first step, under which the item before is finished, ends without a flush");

// Blocks of 8 key columns (bit b: columns [8 b, 8 b + 8) of a step) whose exponentials come from a polynomial on the
// FMA pipe instead of the special-function unit, which at 16 results per clock per SM would otherwise set the pace.
// The polynomial costs more instructions and more energy, and the long launches run at the card's power limit, so the
// choice that takes the fewest clocks gains least.  Two blocks and no more: the polynomial's error (7.5e-5) vanishes in the rounding of
// the probabilities to bf16, but not in the sum of the unrounded ones behind the log-sum-exp (7.2e-5 where one key of such a block
// takes the whole softmax), and every further block adds to it.  A third block (4, 9 and 12 instead of 6 and 13) is not worth that:
// 10 frames of 1,374 tokens, a quarter retained, 269.8 us against 271.8; 100 frames 22.20 ms against 22.54, dense 81.1 against 82.9; frame
// attention of 10 frames 118.1 us against 119.7.
#ifndef AVGGT_POLY_BLOCKS
#define AVGGT_POLY_BLOCKS 0x2040
#endif
constexpr uint32_t kPolyBlocks = AVGGT_POLY_BLOCKS;

struct AttnArgs {
  Plan pl;
  Divisor by_pairs, by_heads, by_window;
  WindowRule rule;
  const float* kmean;   // [H, d] or null
  const float* vmean;
  __nv_bfloat16* O;     // [n_tok, H, d]
  float* lse;           // [n_tok, H] or null
  const int32_t* slot_of_token;   // caller-chosen retained set: compact position of every token, -1 = dropped; else null
  uint32_t* status;     // 4 words
  int32_t frame_mode;   // 0: subsampled global attention over the compact keys.  1: frame attention (Sec. 4.2):
                        //    every frame is a problem of its own, keys and values are the frame's own rows of K and V
  int64_t n_keys;       // keys of one problem: M, or the tokens of a frame
  int32_t n_kv_tiles;   // ceil(n_keys / kTileKV)
  int32_t last_tile_keys;   // keys of a ragged last tile, else 0
  int32_t n_work;       // work items (pairs of query tiles x heads x problems) of the launch; a CTA takes the items
                        // blockIdx.x, blockIdx.x + gridDim.x, ...
  int32_t item_rows;    // query rows of a work item: 256 (two full tiles), or fewer, spread over both tiles
  int32_t split_rows[2], split_lanes[2];   // rows of tile 0 and lanes left free in tile 1: of a work item, of a ragged one
  int32_t pairs;        // work items of one problem and head (kShortLast: the full ones)
  int32_t n_problems;   // kShortLast: problems x heads
  int32_t window;       // kShortLast: so many of them make a window of the numbering (work_item)
  int32_t ragged_rows;  // kShortLast: query rows of a problem's last item, 0 if it is a full one
  int32_t use_diag;     // diag on and |D| > 0
  int32_t use_mean;     // mean_fill on and |D| > 0
  float scale_log2;     // softmax scale * log2(e)
  float inv_scale_log2;
  float poly_range;     // raw score units from kLookBelow to the threshold of a rescale
  float poly_floor;     // the raw score of kPolyFloor
  float log2_count[2];  // log2 weight of the mean column for a retained and for a dropped query (0: unit weight; -inf: absent)
};

// Records of work items (ItemInfo): so many that one is never overwritten while a warp may still read it.  When the producer writes
// the record of item n, q_empty says of item n - 2 and each tile: if the tile is at work in it, its Q K^T have all completed, so that its softmax
// warps have read the scores of its item before that and, with one step per item, may still be before the epilogue of the one
// before (n - 4 at the earliest: the epilogue does not wait behind items that the tile sits out); if it sits the item out, that
// its softmax warps have read the record (sat_out).  (With a barrier of all softmax warps for every record, which says it of each item
// alike, frame attention of 10 frames took 121.5 us instead of 118.1, of 500 frames of 101 tokens 126.4 instead of 120.9.)
constexpr int kInfos = 8;

// Ordered by the arrivals that a phase counts, so that as many threads can initialise them at once (init_barriers).
struct __align__(8) Barriers {
  // one arrival
  uint64_t q_full[2];          // producer -> MMA: the work item's Q tiles are in shared memory (items take the two places in turn)
  uint64_t k_full[kStages], v_full[kStages];
  uint64_t s_full[kQTiles];    // MMA -> softmax: S_t(j) is in tensor memory
  uint64_t o_done[kQTiles][2]; // MMA -> softmax: P_t(j) V_j has completed; even and odd steps apart, since the softmax learns of
                               // P V of step j-2 from the scores of step j only, and of later ones here
  uint64_t info_full[kInfos];  // producer -> softmax: the item's record is in shared memory
  uint64_t own_full;           // producer -> softmax: the item's own rows of K and V and the mean pair are in shared memory
  uint64_t mma_idle[kQTiles];  // MMA issuer t -> itself: every tcgen05.mma it issued has completed
  // one of each tile's issuer
  uint64_t k_empty[kStages], v_empty[kStages];
  // one of each of a tile's softmax warps
  uint64_t o_free[kQTiles];    // softmax -> MMA: O_t of the finished work item has been read out
  uint64_t s_free[kQTiles];    // softmax -> MMA: S_t(j) has been read into registers
  uint64_t p_full[kQTiles][2]; // softmax -> MMA: P_t(j) stored (and O_t rescaled); even and odd steps apart, since a warp may
                               // have finished a step before another warp of its tile has finished the step before
  uint64_t sat_out[2];         // softmax -> MMA: the warp has read the record of an item that its tile sits out; even and odd items apart,
                               // since a warp may have read the next one before another warp has read this one
  // one of each softmax warp
  uint64_t own_empty;          // softmax -> producer: its epilogue has read the own rows
  // of the issuers, where there are keys, and with extra columns of the softmax warps
  uint64_t q_empty[2];         // MMA issuers -> producer: every Q K^T of the work item has completed; with extra columns, softmax ->
                               // producer as well: the epilogue has read Q.  Q may be overwritten
  uint32_t tmem_base;
  uint32_t abort_flag;
};
// A thread each: one thread alone takes 400 clocks for them.
template <bool kExtra>
__device__ __forceinline__ void init_barriers(Barriers* bars, const AttnArgs& a, int tid) {
  constexpr int kSize = sizeof(uint64_t);
  constexpr int kTwo = offsetof(Barriers, k_empty) / kSize, kTile = offsetof(Barriers, o_free) / kSize,
                kAll = offsetof(Barriers, own_empty) / kSize, kQ = offsetof(Barriers, q_empty) / kSize;
  static_assert(kAll + 1 == kQ && kQ + 2 == offsetof(Barriers, tmem_base) / kSize, "order of the barriers");
  if (tid < kQ + 2) {
    const uint32_t count = tid < kTwo ? 1 : tid < kTile ? kQTiles : tid < kAll ? kSoftmaxWarps / kQTiles : tid < kQ ? kSoftmaxWarps
                           : (a.n_kv_tiles > 0 ? kQTiles : 0) + (kExtra ? kSoftmaxWarps : 0);
    mbar_init(smem_u32(bars) + tid * kSize, count);
    fence_mbar_init();
  }
  if (tid == 0) bars->abort_flag = 0;
}

__device__ __forceinline__ void report_timeout(const AttnArgs& a, Barriers* bars, uint32_t where, uint32_t iter) {
  if (atomicCAS(a.status, 0u, 1u) == 0u) {
    a.status[1] = blockIdx.x;
    a.status[2] = where;
    a.status[3] = iter;
  }
  *reinterpret_cast<volatile uint32_t*>(&bars->abort_flag) = 1u;
}

// Bounded wait.  Returns false when the time limit ran out (the failure is
// recorded and the CTA-wide abort flag raised) or when another role aborted.
__device__ __forceinline__ bool wait_bar(uint64_t* bar, uint32_t parity, Barriers* bars, const AttnArgs& a,
                                         uint32_t where, uint32_t iter, bool check_abort = true) {
  const uint32_t b = smem_u32(bar);
  if (mbar_try_wait(b, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (true) {
    if (mbar_try_wait(b, parity)) return true;
    if ((++spins & 0xffu) == 0) {
      if (check_abort && *reinterpret_cast<volatile uint32_t*>(&bars->abort_flag)) return false;
      if (globaltimer_ns() - t0 > AVGGT_WAIT_LIMIT_NS) {
        report_timeout(a, bars, where, iter);
        return false;
      }
    }
  }
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// Register budget per thread after the roles have split.  The sum over all warps must not
// exceed what the launch allocated (96 x 640): a setmaxnreg.inc that asks for more than the
// pool can ever hold waits for ever, and that wait has no time limit.
constexpr int kRegsLaunch = 96;   // 65536 / 640 threads, rounded down to the allocation unit
constexpr int kRegsSoftmax = 112, kRegsOther = 32;
static_assert(kRegsSoftmax * kSoftmaxWarps + kRegsOther * (kThreads / 32 - kSoftmaxWarps) <= kRegsLaunch * (kThreads / 32),
              "register budget after setmaxnreg exceeds the launch allocation");

// A work item.
struct WorkItem {
  int head;
  int key_row0;   // frame attention: token index of the frame's first key
  int row0;       // first query row (token index)
  int64_t end;    // one past the item's last query row
  int split;      // 0: item of item_rows rows, 1: ragged one
};
// One of its query tiles.
struct QueryTile {
  int q0;         // token index of lane 0 (negative where the lanes before `first` reach back that far)
  int first;      // query rows [first, last) are wanted
  int64_t last;
};

// Where an item stands in the numbering of kShortLast.
struct Place {
  uint32_t problem0;   // first problem (x heads) of the item's window
  uint32_t n;          // the item's number in the window
  uint32_t n_full;     // full items of the window; the ragged ones follow
};
__device__ __forceinline__ Place place_of(const AttnArgs& a, uint32_t item) {
  Place p;
  p.problem0 = divide(item, a.by_window, p.n) * a.window;
  const uint32_t left = a.n_problems - p.problem0;
  p.n_full = (left < static_cast<uint32_t>(a.window) ? left : a.window) * a.pairs;
  return p;
}

// Items are numbered with the pair of query tiles fastest, then the head, then (frame
// attention) the frame, so that the CTAs running side by side share one head's keys in L2.  kShortLast (launches without the
// extra columns, i.e. frame attention, and the dense layer, where it makes no difference): the ragged last items come after the
// full ones of their window of the numbering (choose_window), so that every CTA meets some (with six items per frame and head and
// 148 CTAs every second CTA never met a short one).  With the trimmed last key tile and one window, frame attention of 10 frames
// 125.3 -> 122.0 us, of 100 frames 1187 -> 1171 us; with tile 1 left out of items of one tile 118.8 and 1139 us (of the same
// run: 124.4 and 1177 before).  The card is at its power limit there, so it is the products not made that count more than
// the balance.
template <bool kShortLast>
__device__ __forceinline__ WorkItem work_item(const AttnArgs& a, uint32_t item) {
  WorkItem w;
  uint32_t qp, head;
  uint32_t rest;
  bool ragged = false;
  if (kShortLast) {
    const Place p = place_of(a, item);
    rest = p.problem0 + divide(p.n, a.by_pairs, qp);
    ragged = p.n >= p.n_full;
    if (ragged) {
      rest = p.problem0 + p.n - p.n_full;
      qp = a.pairs;
    }
  } else {
    rest = divide(item, a.by_pairs, qp);
  }
  const uint32_t frame = divide(rest, a.by_heads, head);
  w.head = static_cast<int>(head);
  w.key_row0 = static_cast<int>(frame) * a.pl.L;   // the subsampled layer has one problem
  w.row0 = w.key_row0 + static_cast<int>(qp) * a.item_rows;
  const int64_t end = a.frame_mode ? static_cast<int64_t>(w.key_row0) + a.pl.L : a.pl.n_tok;
  w.end = end - w.row0 > a.item_rows ? static_cast<int64_t>(w.row0) + a.item_rows : end;
  w.split = kShortLast ? (ragged ? 1 : 0) : (end - w.row0 < a.item_rows ? 1 : 0);
  return w;
}

// An item of fewer than 256 rows is cut in two halves by groups of 16 rows (one softmax warp), the second half in the upper lanes
// of its tile: the warps with work are spread over the four schedulers, and both tiles' products overlap.  Warps without rows
// compute nothing.
//
// kShortLast: a last item of one tile is left to tile 0, and tile 1 sits it out, products and all.  (The subsampled layer meets
// such an item once per head, or is so small that nothing but latency counts; there the halves are as good and the code simpler.)
__device__ __forceinline__ QueryTile query_tile(const AttnArgs& a, const WorkItem& w, int t) {
  QueryTile q;
  const int cut = w.row0 + a.split_rows[w.split];   // first row of tile 1
  q.first = t == 0 ? w.row0 : cut;
  q.q0 = t == 0 ? w.row0 : cut - a.split_lanes[w.split];
  q.last = t == 0 && cut < w.end ? cut : w.end;
  return q;
}

// What the softmax warps need to know of a work item: found once, by the producer (sixteen warps that each found it for themselves,
// at the start and again in the epilogue, spent some 150 instructions a time on it).
struct ItemInfo {
  int head;
  int active[kQTiles];   // the tile takes part in the item
  int q0[kQTiles], first[kQTiles], last[kQTiles];   // QueryTile
};

struct SmemLayout {
  uint8_t* q;   // 2 places of kQTiles tiles
  uint8_t* k;   // kStages tiles
  uint8_t* v;   // kStages tiles
  uint8_t* own_v;   // kQTiles tiles: V of the query rows; the epilogue turns O around here, each warp in its own rows
  uint8_t* own_k;   // kQTiles tiles: K of the query rows (with extra columns only, as what follows)
  float* means;     // the head's mean Key and mean Value
  uint8_t* ones;   // 16 rows of 64 values: 1 in column 0, else 0 (ones_block)
};

// The producer and the MMA issuers run with all 32 lanes of their warp in step (every branch
// condition is made warp-uniform with a vote) and issue the TMA / tcgen05 instructions from one
// elected lane.  Those instructions take their operands from the uniform datapath; issued from
// divergent single-lane code they fall on a slow path that costs on the order of 100 clocks each.
constexpr uint32_t kFullMask = 0xffffffffu;

__device__ __forceinline__ bool wait_bar_warp(uint64_t* bar, uint32_t parity, Barriers* bars, const AttnArgs& a,
                                              uint32_t where, uint32_t iter, bool check_abort = true) {
  return __all_sync(kFullMask, wait_bar(bar, parity, bars, a, where, iter, check_abort));
}

// kShortLast: tile 1 has rows in the item
__device__ __forceinline__ bool tile_has_rows(const AttnArgs& a, uint32_t item) {
  if (a.item_rows <= kTileQ) return false;
  if (a.ragged_rows == 0 || a.ragged_rows > kTileQ) return true;
  const Place p = place_of(a, item);
  return p.n < p.n_full;
}

// ------------------------------------------------------------------ TMA producer (one warp)
template <bool kShortLast>
__device__ __forceinline__ void producer_role(const CUtensorMap* tm_q, const CUtensorMap* tm_k, const CUtensorMap* tm_v,
                                              const CUtensorMap* tm_own_k, const CUtensorMap* tm_own_v, const AttnArgs& a, Barriers* bars,
                                              ItemInfo* infos, const SmemLayout& sm, WorkItem wi, QueryTile tile0, QueryTile tile1) {
  constexpr bool kExtra = !kShortLast;
  const int n_kv = a.n_kv_tiles;   // 0 where there are no retained keys
  int k_issued = 0, v_issued = 0;   // K / V copies issued so far, over all work items
  int stage = 0;
  uint32_t empty_parity = 1;   // a fresh barrier passes the wait on the "previous" phase at once
  bool ok = true;
  int n_done = 0;              // work items completed by this role
  int q_issued = 0;            // work items whose Q copies have been issued
  int own_issued = 0;          // ... whose own rows' copies have been issued
  for (uint32_t item = blockIdx.x; item < static_cast<uint32_t>(a.n_work) && ok; item += gridDim.x, ++n_done) {
    const uint32_t failed = *reinterpret_cast<volatile uint32_t*>(a.status);
    if (n_done > 0) {
      wi = work_item<kShortLast>(a, item);
      tile0 = query_tile(a, wi, 0);
      tile1 = query_tile(a, wi, 1);
    }
    const int head = wi.head;
    const int place = n_done & 1;
    const QueryTile tile[kQTiles] = {tile0, tile1};
    // the Q tiles of the work item before the last one are no longer read by any Q K^T
    ok = wait_bar_warp(&bars->q_empty[place], ((n_done >> 1) & 1) ^ 1, bars, a, 14, n_done);
    if (!ok) break;
    if (elect_one()) {
      const uint32_t qb = smem_u32(&bars->q_full[place]);
      mbar_arrive_expect_tx(qb, kQTiles * kTileBytes);
#pragma unroll
      for (int t = 0; t < kQTiles; ++t)
        tma_load_2d(smem_u32(sm.q + (place * kQTiles + t) * kTileBytes), tm_q, head * kHeadDim, tile[t].q0, qb);
    }
    __syncwarp();
    ++q_issued;
    // A wait has run out in another thread block (or had before this one began): the launch is abandoned.  Looked at here because
    // the word takes some 700 clocks to come, which a launch of a single item would wait for.
    if (__any_sync(kFullMask, failed != 0u)) {
      *reinterpret_cast<volatile uint32_t*>(&bars->abort_flag) = 1u;
      ok = false;
      break;
    }
    if (elect_one()) {
      ItemInfo& info = infos[n_done % kInfos];
      info.head = head;
      info.active[0] = 1;
      info.active[1] = kExtra || tile_has_rows(a, item) ? 1 : 0;
#pragma unroll
      for (int t = 0; t < kQTiles; ++t) {
        info.q0[t] = tile[t].q0;
        info.first[t] = tile[t].first;
        info.last[t] = static_cast<int>(tile[t].last);
      }
      mbar_arrive(smem_u32(&bars->info_full[n_done % kInfos]));
    }
    __syncwarp();
    for (int it = 0; it < n_kv; ++it) {
      ok = wait_bar_warp(&bars->k_empty[stage], empty_parity, bars, a, 10, it);
      if (!ok) break;
#ifdef AVGGT_TEST_SKIP_K_LOAD
      // Build for the wait-limit test only (never part of libavggt.so): the first thread block leaves out one K
      // tile, so that the waits on it run out, the block reports the time-out and every role leaves in order.
      const bool skip_load = it == AVGGT_TEST_SKIP_K_LOAD && n_done == 0 && blockIdx.x == 0;
#else
      constexpr bool skip_load = false;
#endif
      if (elect_one() && !skip_load) {
        const uint32_t kb = smem_u32(&bars->k_full[stage]);
        mbar_arrive_expect_tx(kb, kKeyTileBytes);
        if (a.frame_mode) tma_load_2d(smem_u32(sm.k + stage * kKeyTileBytes), tm_k, head * kHeadDim, wi.key_row0 + it * kTileKV, kb);
        else tma_load_3d(smem_u32(sm.k + stage * kKeyTileBytes), tm_k, 0, it * kTileKV, head, kb);
      }
      __syncwarp();
      ++k_issued;
      ok = wait_bar_warp(&bars->v_empty[stage], empty_parity, bars, a, 11, it);
      if (!ok) break;
      if (elect_one()) {
        const uint32_t vb = smem_u32(&bars->v_full[stage]);
        mbar_arrive_expect_tx(vb, kKeyTileBytes);
        if (a.frame_mode) tma_load_2d(smem_u32(sm.v + stage * kKeyTileBytes), tm_v, head * kHeadDim, wi.key_row0 + it * kTileKV, vb);
        else tma_load_3d(smem_u32(sm.v + stage * kKeyTileBytes), tm_v, 0, it * kTileKV, head, vb);
      }
      __syncwarp();
      ++v_issued;
      if (++stage == kStages) { stage = 0; empty_parity ^= 1; }
    }
    // The query rows' own K and V and the mean pair, which the epilogue of the item before has to have read: it comes after this
    // item's first step, whose keys and values are on their way.
    if (kExtra && ok) {
      ok = wait_bar_warp(&bars->own_empty, (n_done & 1) ^ 1, bars, a, 15, n_done);
      if (!ok) break;
      if (elect_one()) {
        const uint32_t ob = smem_u32(&bars->own_full);
        constexpr uint32_t kMeanBytes = kHeadDim * sizeof(float);
        mbar_arrive_expect_tx(ob, (a.use_diag ? 2 * kQTiles * kTileBytes : 0) + (a.use_mean ? 2 * kMeanBytes : 0));
        if (a.use_diag) {
#pragma unroll
          for (int t = 0; t < kQTiles; ++t) {
            tma_load_2d(smem_u32(sm.own_k + t * kTileBytes), tm_own_k, head * kHeadDim, tile[t].q0, ob);
            tma_load_2d(smem_u32(sm.own_v + t * kTileBytes), tm_own_v, head * kHeadDim, tile[t].q0, ob);
          }
        }
        if (a.use_mean) {
          bulk_load(smem_u32(sm.means), a.kmean + head * kHeadDim, kMeanBytes, ob);
          bulk_load(smem_u32(sm.means + kHeadDim), a.vmean + head * kHeadDim, kMeanBytes, ob);
        }
      }
      __syncwarp();
      ++own_issued;
    }
  }
  if (!ok) {
    // let the copies still in flight land before the CTA gives up its shared memory: the Q tiles of the last two work
    // items begun, the last own rows, and the last kStages issued into either ring (earlier ones completed before their stage was reused)
    for (int back = 1; back <= 2; ++back) {
      const int jq = q_issued - back;
      if (jq >= 0) (void)wait_bar_warp(&bars->q_full[jq & 1], (jq >> 1) & 1, bars, a, 12, jq, false);
    }
    if (own_issued > 0) (void)wait_bar_warp(&bars->own_full, (own_issued - 1) & 1, bars, a, 16, own_issued, false);
    for (int back = 1; back <= kStages; ++back) {
      const int jk = k_issued - back, jv = v_issued - back;
      if (jk >= 0) (void)wait_bar_warp(&bars->k_full[jk % kStages], (jk / kStages) & 1, bars, a, 12, jk, false);
      if (jv >= 0) (void)wait_bar_warp(&bars->v_full[jv % kStages], (jv / kStages) & 1, bars, a, 13, jv, false);
    }
  }
}

// ------------------------------------------------------------------ MMA issuer (one warp per query tile)
// Per tile the order of events is fixed: S_t(j) is read by the softmax (s_free) before P_t(j) is
// stored (p_full), which precedes the read of S_t(j+1).  The issuer of tile t therefore waits, in
// turn, for "S_t(j) read and K_{j+1} loaded" -> Q K^T of step j+1 (or of step 0 of the next work
// item), then "P_t(j) stored and V_j loaded" -> P V of step j.  S_t(j+1) overwrites P_t(j-1) and part of S_t(j): the tensor core takes
// a thread's products in the order they were issued, and P V of step j-1 was issued before.
// A K or V stage is released when both tiles' issuers have committed
// their product on it (the empty barriers count two arrivals).
//
// The issuing is on the chain from the slowest warp of a step to the next scores, and it shares its scheduler with four softmax
// warps, so each instruction of it counts: the lower halves of the operand descriptors advance by additions of a constant, the
// upper halves are constants, and of several waits the one that is satisfied last comes last.
template <int t>
__device__ __forceinline__ void issue_qk(Barriers* bars, uint32_t tmem, uint32_t desc_q, uint32_t desc_k, int stage, bool odd,
                                         uint32_t idesc) {
  if (elect_one()) {
    const uint32_t d = tmem + t * kTmemTileStride + (odd ? kColSOdd : 0);
#pragma unroll
    for (int k = 0; k < kHeadDim / 16; ++k) umma_ss_lo(d, desc_q + (k * 32 >> 4), desc_k + (k * 32 >> 4), idesc, k > 0);
    umma_commit(smem_u32(&bars->s_full[t]));
    umma_commit(smem_u32(&bars->k_empty[stage]));
  }
  __syncwarp();
}

// O_t += P_t V and, as columns 64..79 of the same product, the row sums of P: the descriptor's leading byte offset leads
// from a slice of 16 keys of the V tile to the ones block, which serves as value columns 64..79 of every slice.
template <int t, bool kTrim>
__device__ __forceinline__ void issue_pv(Barriers* bars, uint32_t tmem, uint32_t desc_v, int stage, bool odd, bool first,
                                         int slices) {
  if (elect_one()) {
    constexpr uint32_t idesc = umma_idesc_bf16(kTileQ, kPvCols, true);
    constexpr uint32_t kSlice = 16 * kHeadDim * 2;   // bytes of 16 keys: the start moves on, the offset to the ones shrinks
    constexpr uint32_t kAdvance = (kSlice >> 4) - ((kSlice >> 4) << 16);
    const uint32_t p = tmem + t * kTmemTileStride + (odd ? kColPOdd : 0);
    umma_ts_lo(tmem + t * kTmemTileStride + kColO, p, desc_v, idesc, !first);
#pragma unroll
    for (int k = 1; k < kTileKV / 16; ++k)
      if (!kTrim || k < slices) umma_ts_lo(tmem + t * kTmemTileStride + kColO, p + k * 8, desc_v + k * kAdvance, idesc, true);
    umma_commit(smem_u32(&bars->o_done[t][odd]));
    umma_commit(smem_u32(&bars->v_empty[stage]));
  }
  __syncwarp();
}

// kTrim: of a ragged last tile compute only as many columns and slices of 16 keys as hold keys.  Worth its instructions where steps
// are few (frame attention of 1,374 tokens has 30 keys in the last of 13 tiles: 1.5 %); in the subsampled layer they cost 1 %.
template <int t, bool kTrim>
__device__ __forceinline__ void mma_issue_loop(const AttnArgs& a, Barriers* bars, const SmemLayout& sm, uint32_t tmem) {
  static_assert(kStages >= 2, "the K ring must hold the tile in use and the next one");
  const int n_kv = a.n_kv_tiles;
  // lower halves of the descriptors (umma_desc_lo)
  const uint32_t q_desc = umma_desc_lo(smem_u32(sm.q) + t * kTileBytes, 16), k_desc = umma_desc_lo(smem_u32(sm.k), 16);
  const uint32_t v_desc = umma_desc_lo(smem_u32(sm.v), smem_u32(sm.ones) - smem_u32(sm.v));
  constexpr uint32_t kStage = kKeyTileBytes >> 4;         // a stage further on the start advances ...
  constexpr uint32_t kStageV = kStage - (kStage << 16);   // ... and the offset to the ones shrinks
  if (n_kv == 0) return;   // no retained keys: the epilogue's two extra columns are the whole layer
  const int ragged_slices = a.last_tile_keys != 0 ? (a.last_tile_keys + 15) >> 4 : kTileKV / 16;
  constexpr uint32_t kDescQk = umma_idesc_bf16(kTileQ, kTileKV, false);
  const uint32_t ragged_desc_qk = umma_idesc_bf16(kTileQ, 16 * ragged_slices, false);

  // Running over all work items of the CTA: the ring positions of the next K and V tile, and g, the number of key
  // steps of this tile so far (the phase of the per-step barriers).
  int k_stage = 0, v_stage = 0;
  uint32_t k_parity = 0, v_parity = 0;   // parity of their "full" phase
  int g = 0;
  int n_done = 0;
  int n_active = 0;          // work items this tile had rows in
  uint32_t sat_out_parity = 0;   // bit of the even, of the odd items
  bool first_issued = false; // Q K^T of the item's first step went out with the item before
  for (uint32_t item = blockIdx.x; item < static_cast<uint32_t>(a.n_work); item += gridDim.x, ++n_done) {
    if (kTrim && t > 0 && !tile_has_rows(a, item)) {
      // the tile sits this item out: pass its tiles on in step
      if (!wait_bar_warp(&bars->q_full[n_done & 1], (n_done >> 1) & 1, bars, a, 20, n_done)) return;
      for (int j = 0; j < n_kv; ++j) {
        if (!wait_bar_warp(&bars->k_full[k_stage], k_parity, bars, a, 24 + t, j)) return;
        if (elect_one()) mbar_arrive(smem_u32(&bars->k_empty[k_stage]));
        __syncwarp();
        if (++k_stage == kStages) { k_stage = 0; k_parity ^= 1; }
        if (!wait_bar_warp(&bars->v_full[v_stage], v_parity, bars, a, 28 + t, j)) return;
        if (elect_one()) mbar_arrive(smem_u32(&bars->v_empty[v_stage]));
        __syncwarp();
        if (++v_stage == kStages) { v_stage = 0; v_parity ^= 1; }
      }
      // Q last: its places pace the producer's records
      if (!wait_bar_warp(&bars->sat_out[n_done & 1], (sat_out_parity >> (n_done & 1)) & 1, bars, a, 21, n_done)) return;
      sat_out_parity ^= 1u << (n_done & 1);
      if (elect_one()) mbar_arrive(smem_u32(&bars->q_empty[n_done & 1]));
      __syncwarp();
      continue;
    }
    const bool more = item + gridDim.x < static_cast<uint32_t>(a.n_work) &&
                      (!kTrim || t == 0 || tile_has_rows(a, item + gridDim.x));
    // j = -1: Q K^T of the first step, where it has not been issued with the item before
    for (int j = first_issued ? 0 : -1; j < n_kv; ++j) {
      const bool last = j + 1 == n_kv;
      if (!last || more) {
        const int next = last ? 0 : j + 1;                  // step within its work item
        const int next_item = last ? n_done + 1 : n_done;
        const int place = next_item & 1;
        if (next == 0 && !wait_bar_warp(&bars->q_full[place], (next_item >> 1) & 1, bars, a, 20, n_done)) return;
        if (!wait_bar_warp(&bars->k_full[k_stage], k_parity, bars, a, 24 + t, g + j)) return;
        if (g + j >= 0 && !wait_bar_warp(&bars->s_free[t], (g + j) & 1, bars, a, 22 + t, g + j)) return;
        tc_fence_after();
        issue_qk<t>(bars, tmem, q_desc + place * (kQTiles * kTileBytes >> 4), k_desc + k_stage * kStage, k_stage, ((g + j + 1) & 1) != 0,
                    kTrim && next + 1 == n_kv ? ragged_desc_qk : kDescQk);
        if (++k_stage == kStages) { k_stage = 0; k_parity ^= 1; }
        if (next + 1 == n_kv) {   // every Q K^T of the work item has been issued: when they have completed, Q may be overwritten
          if (elect_one()) umma_commit(smem_u32(&bars->q_empty[place]));
          __syncwarp();
        }
      }
      if (j < 0) continue;
      if (!wait_bar_warp(&bars->v_full[v_stage], v_parity, bars, a, 28 + t, g + j)) return;
      // the first P V of a work item overwrites O_t: the previous item's epilogue must have read it out
      if (j == 0 && n_active > 0 && !wait_bar_warp(&bars->o_free[t], (n_active - 1) & 1, bars, a, 29, n_done)) return;
      if (!wait_bar_warp(&bars->p_full[t][(g + j) & 1], ((g + j) >> 1) & 1, bars, a, 26 + t, g + j)) return;
      tc_fence_after();
      issue_pv<t, kTrim>(bars, tmem, v_desc + v_stage * kStageV, v_stage, ((g + j) & 1) != 0, j == 0, last ? ragged_slices : kTileKV / 16);
      if (++v_stage == kStages) { v_stage = 0; v_parity ^= 1; }
    }
    first_issued = more;
    g += n_kv;
    ++n_active;
  }
}

// The issue loop, then (on every path out of it, a wait that ran out included) a wait until the
// tensor core has finished everything this warp issued: the CTA must not free its tensor memory
// or leave its shared memory while a tcgen05.mma still reads or writes them.
template <int t, bool kTrim>
__device__ __forceinline__ void mma_role(const AttnArgs& a, Barriers* bars, const SmemLayout& sm, uint32_t tmem) {
  mma_issue_loop<t, kTrim>(a, bars, sm, tmem);
  __syncwarp();
  if (elect_one()) umma_commit(smem_u32(&bars->mma_idle[t]));
  __syncwarp();
  (void)wait_bar_warp(&bars->mma_idle[t], 0, bars, a, 70 + t, 0, false);
}

// ------------------------------------------------------------------ softmax warpgroup (128 threads per tile)
// 2^x for a pair of values on the FMA pipe.  x = n + r with n = round(x), |r| <= 1/2: adding
// 1.5 * 2^23 leaves n in the low mantissa bits of the sum; 2^r is a degree-3 minimax polynomial
// (relative error 7.5e-5, a twenty-sixth of the bf16 rounding step the result goes through);
// 2^n is applied by adding n to the exponent field.  Valid for -126 <= x <= 100; the caller sees to that.
__device__ __forceinline__ void exp2_poly_pair(uint64_t x2, float& p0, float& p1) {
  const uint64_t magic = pack_f32x2(12582912.0f, 12582912.0f);
  const uint64_t t = add_f32x2(x2, magic);
  const uint64_t r = sub_f32x2(x2, sub_f32x2(t, magic));
  uint64_t q = fma_f32x2(pack_f32x2(0x1.c3f76p-5f, 0x1.c3f76p-5f), r, pack_f32x2(0x1.f0de1ap-3f, 0x1.f0de1ap-3f));
  q = fma_f32x2(q, r, pack_f32x2(0x1.62f31ap-1f, 0x1.62f31ap-1f));
  q = fma_f32x2(q, r, pack_f32x2(0x1.fff692p-1f, 0x1.fff692p-1f));
  float t0, t1, q0, q1;
  unpack_f32x2(t, t0, t1);
  unpack_f32x2(q, q0, q1);
  p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
  p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}
// A step looks at its rows (softmax_step) when one of its scores lies more than so many log2 units below the reference, and gives
// those more than kPolyLowest below a score that comes out of the polynomial as 2^-122.  Above it the polynomial is right, down
// to -126.5.  The look is decided on raw scores, whose rounding shifts it by up to |m| 2^-20 log2 units at a reference m: less
// than the one unit between the two for |m| < kLargeReference.  A row with a larger reference looks at every step.
constexpr float kLookBelow = -125.0f, kPolyLowest = -126.0f;
constexpr float kLargeReference = 1048576.0f;
// That score, in log2 units: so far below any reference that it does not matter which, and beyond 2^48, where the polynomial finds
// r = 0 and takes the exponent from the lowest bits of x: 390 of 512 is -122 (within 2, for the roundings of the raw score,
// its product with the scale and the reference).  A score raised to the polynomial's range by its raw value, as one would, misses that
// range for |m| > 2^23, where the raw scores are further apart.
constexpr float kPolyFloor = -0x1.00030cp80f;

// What a softmax thread knows about itself.  A softmax warp works on 16 query rows of its tile, all columns
// of a key step: the tensor-memory lanes [32 q + 16 h, 32 q + 16 h + 16) of the tile.  Its tensor-memory
// accesses use the 16-lane shapes, which spread a row over the four threads of a quad: thread `lane` holds,
// of every block of 8 columns, columns 2 i and 2 i + 1 (i = lane % 4) of the rows lane / 4 and lane / 4 + 8.
// A row's maximum therefore takes two shuffles within the quad and no shared memory, and every row
// is handled inside one warp.
struct SoftmaxThread {
  int t;        // query tile of the CTA
  int h;        // which 16 of the 32 lanes of the warp's tensor-memory quarter
  int q;        // tensor-memory quarter (and scheduler): lanes [32 q, 32 q + 32)
  int lane;
  uint32_t base;   // tensor-memory address of the tile's columns, first lane of the warp's 16
};

// tensor memory <-> registers in the 16-lane shapes (layout above): S, O and the row sums as 32-bit columns, P as
// columns of bf16 pairs
__device__ __forceinline__ void tmem_ld_rows16_c8(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_rows16_c8(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.16x256b.x1.b32 [%0], {%1, %2, %3, %4};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}
// the 112 score columns of a step in three pieces: 64, 32 and 16
__device__ __forceinline__ void tmem_ld_rows16_scores(uint32_t taddr, uint32_t (&r)[4 * kBlocks]) {
  static_assert(kTileKV == 112, "three pieces");
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
        "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47])
      : "r"(taddr + 64)
      : "memory");
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55])
               : "r"(taddr + 96)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_rows16_c32(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_rows16_c32(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x4.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
// bf16 pairs of 4 blocks of 8 keys: register 2 n + hi -> row hi of the thread, pair column 4 n + i
__device__ __forceinline__ void tmem_st_rows16_p16(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

__device__ __forceinline__ void tmem_st_rows16_p8(uint32_t taddr, const uint32_t (&r)[8]) {   // of 2 blocks
  asm volatile("tcgen05.st.sync.aligned.16x128b.x2.b32 [%0], {%1, %2, %3, %4};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
               : "memory");
}

// value over the four threads of a quad
__device__ __forceinline__ float quad_max(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2));
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}

// Running state of the thread's two rows (the same in all four threads of a quad, except the partial sums).
struct RowState {
  float neg_m[2];         // minus the reference maximum of the stored exponentials (log2 units); +inf before the first tile
  float look_above[2];    // raw score above which the reference may have to move; -inf before the first tile
  float l_exact[2];       // this thread's part of the sum of the unrounded 2^(scale_log2 * s - m): log-sum-exp output only
};

// Blocks 4 kGroup .. of the thread's scores of a key step (register 4 b + 2 hi + e: row hi, column 8 b + 2 i + e) -> bf16
// probabilities relative to the rows' reference maxima; kLse: adds the unrounded ones to sum_exact2.  Written pair by pair in
// dependency order; the instruction scheduler interleaves the pairs.
template <int kGroup, bool kMasked, bool kLse, uint32_t kPoly>
__device__ __forceinline__ void exp_group(const uint32_t (&s)[4 * kBlocks], const RowState& st, uint64_t scale2,
                                          uint64_t (&sum_exact2)[2], uint32_t (&pk)[8], int n_blocks) {
#pragma unroll
  for (int n = 0; n < 4; ++n) {
    const int b = 4 * kGroup + n;
    if (b >= kBlocks) break;
    // ragged last step: a block of 8 columns with no key in it gives zeros without any arithmetic
    if (kMasked && b >= n_blocks) {
      pk[2 * n] = 0u;
      pk[2 * n + 1] = 0u;
      continue;
    }
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      const int c = 4 * b + 2 * hi;
      const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(s[c]), __uint_as_float(s[c + 1])), scale2,
                                    pack_f32x2(st.neg_m[hi], st.neg_m[hi]));
      float p0, p1;
      if ((kPoly >> b) & 1) {
        exp2_poly_pair(x2, p0, p1);
      } else {
        float x0, x1;
        unpack_f32x2(x2, x0, x1);
        p0 = ex2_approx(x0);
        p1 = ex2_approx(x1);
      }
      pk[2 * n + hi] = pack_bf16x2(p0, p1);
      if (kLse) sum_exact2[hi] = add_f32x2(sum_exact2[hi], pack_f32x2(p0, p1));
    }
  }
}

// One step of the online softmax of the thread's two rows: S_t(j) in tensor memory -> P_t(j) in tensor
// memory, running reference maxima updated.
//
// The 56 scores are pulled into registers at once and the warp's share of S_t is released, so that the next
// Q K^T runs under this step's exponentials.  What the step does next depends on the row maxima only when one of them is
// far above its reference (lazy rescale: more than 2^8), so the first group of exponentials is computed against the old
// references while the maxima are being taken, and the common case ends in one vote: no shuffles, no wait for the previous
// P V (P has a place of its own in alternate steps).  The other case moves the references (a row decides by its own maximum,
// so its bits do not depend on its neighbours), rescales O and the row sums, replaces the scores that lie below the range of
// the polynomial, and computes the first group again.  The vote compares raw scores with a limit that errs towards looking;
// what to do is then decided in log2 units, where a large reference costs no more than its own rounding.
// Measured with the tensor core in the loop but without memory traffic, for 2 tiles x 128 keys on one SM: 2270 clocks
// with the maxima shuffled, the sums taken by the softmax warps and a wait for P V in every step, 1990 without those
// waits and sums, 1860 with the vote instead of the shuffles, 1740 with the first group ahead of it, 1695 with the range check
// of the polynomial in the same vote instead of a clamp per score.
//
// gj: this tile's key steps so far, over all work items of the CTA.  kPoly: blocks of 8 columns
// whose exponentials are polynomials.  kLse: also keep the sum of the unrounded exponentials, for the
// log-sum-exp output.  kMasked: columns >= valid are excluded.
template <bool kMasked, bool kLse, uint32_t kPoly>
__device__ __forceinline__ bool softmax_step(const SoftmaxThread& me, int gj, int valid, RowState& st, Barriers* bars,
                                             const AttnArgs& a) {
  const bool odd = (gj & 1) != 0;
  const uint32_t tP = me.base + (odd ? kColPOdd : 0);
  if (!wait_bar(&bars->s_full[me.t], gj & 1, bars, a, 40 + me.t, gj)) return false;
  tc_fence_after();
  uint32_t s[4 * kBlocks];
  tmem_ld_rows16_scores(me.base + (odd ? kColSOdd : 0), s);
  tmem_wait_ld();     // for the whole warp: one lane may speak for it
  tc_fence_before();
  // (elected rather than lane 0: a branch on the lane number costs a reconvergence, 4 % of a ten-frame layer)
  if (elect_one()) mbar_arrive(smem_u32(&bars->s_free[me.t]));

  if (kMasked) {
#pragma unroll
    for (int c = 0; c < 4 * kBlocks; ++c)
      if (8 * (c >> 2) + 2 * (me.lane & 3) + (c & 1) >= valid) s[c] = __float_as_uint(-INFINITY);
  }
  const int n_blocks = kMasked ? (valid + 7) >> 3 : kBlocks;   // blocks of 8 columns that hold a key
  const uint64_t scale2 = pack_f32x2(a.scale_log2, a.scale_log2);
  uint64_t sum_exact2[2] = {pack_f32x2(0.f, 0.f), pack_f32x2(0.f, 0.f)};
  uint32_t pk[8];   // P of 32 keys x 2 rows as bf16 pairs
  constexpr bool kAhead = !kLse && !kMasked;   // first group before the vote
  if (kAhead) exp_group<0, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);

  float mx[2], mn[2];
  bool look = false;
#pragma unroll
  for (int hi = 0; hi < 2; ++hi) {
    float x = fmaxf(__uint_as_float(s[2 * hi]), __uint_as_float(s[2 * hi + 1]));
    float y = fmaxf(__uint_as_float(s[2 * kBlocks + 2 * hi]), __uint_as_float(s[2 * kBlocks + 2 * hi + 1]));
#pragma unroll
    for (int b = 1; b < kBlocks / 2; ++b) {
      x = max3(x, __uint_as_float(s[4 * b + 2 * hi]), __uint_as_float(s[4 * b + 2 * hi + 1]));
      y = max3(y, __uint_as_float(s[2 * kBlocks + 4 * b + 2 * hi]), __uint_as_float(s[2 * kBlocks + 4 * b + 2 * hi + 1]));
    }
    mx[hi] = fmaxf(x, y);
    mn[hi] = INFINITY;
#pragma unroll
    for (int b = 0; b < kBlocks; ++b)
      if ((kPoly >> b) & 1) mn[hi] = min3(mn[hi], __uint_as_float(s[4 * b + 2 * hi]), __uint_as_float(s[4 * b + 2 * hi + 1]));
    look = look || mx[hi] > st.look_above[hi] || (kPoly != 0 && mn[hi] < st.look_above[hi] - a.poly_range);
  }
  if (__any_sync(0xffffffffu, look)) {
    float alpha[2];
    bool jump_any = false;
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      const float m = quad_max(mx[hi]) * a.scale_log2;
      alpha[hi] = 1.0f;
      if (m > kRescaleThreshold - st.neg_m[hi]) {
        jump_any = jump_any || st.neg_m[hi] != INFINITY;   // nothing to rescale on the first tile
        alpha[hi] = ex2_approx(-m - st.neg_m[hi]);
        st.neg_m[hi] = -m;
        // less what the roundings on the way to this limit and to the next m can amount to
        st.look_above[hi] = fabsf(m) < kLargeReference
                                ? (m + kRescaleThreshold - (fabsf(m) + kRescaleThreshold) * 0x1p-21f) * a.inv_scale_log2
                                : -INFINITY;
        if (kLse) st.l_exact[hi] *= alpha[hi];
      }
    }
    if (__any_sync(0xffffffffu, jump_any)) {
      // O_t must be at rest
      if (!wait_bar(&bars->o_done[me.t][!odd], ((gj - 1) >> 1) & 1, bars, a, 30 + me.t, gj)) return false;
      tc_fence_after();
      // the warp's 16 rows of the accumulator, 32 columns at a time (register 4 b + 2 hi + e is row hi): with the scores in
      // registers there is no room for more
#pragma unroll 1
      for (int half = 0; half < 2; ++half) {
        uint32_t o[16];
        tmem_ld_rows16_c32(me.base + kColO + 32 * half, o);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 16; ++c) o[c] = __float_as_uint(__uint_as_float(o[c]) * alpha[(c >> 1) & 1]);
        tmem_st_rows16_c32(me.base + kColO + 32 * half, o);
      }
      uint32_t l[4];
      tmem_ld_rows16_c8(me.base + kColL, l);
      tmem_wait_ld();
#pragma unroll
      for (int c = 0; c < 4; ++c) l[c] = __float_as_uint(__uint_as_float(l[c]) * alpha[c >> 1]);
      tmem_st_rows16_c8(me.base + kColL, l);
    }
    if (kPoly != 0) {
#pragma unroll
      for (int c = 0; c < 4 * kBlocks; ++c)
        if (((kPoly >> (c >> 2)) & 1) && fmaf(__uint_as_float(s[c]), a.scale_log2, st.neg_m[(c >> 1) & 1]) < kPolyLowest)
          s[c] = __float_as_uint(a.poly_floor);
    }
    if (kAhead) exp_group<0, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);
  }

  // exponentials, rounded to bf16 for the value product (whose column of ones sums the rounded values, so that numerator
  // and denominator carry the same weights)
  if (!kAhead) exp_group<0, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);
  tmem_st_rows16_p16(tP, pk);
  exp_group<1, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);
  tmem_st_rows16_p16(tP + 16, pk);
  exp_group<2, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);
  tmem_st_rows16_p16(tP + 32, pk);
  exp_group<3, kMasked, kLse, kPoly>(s, st, scale2, sum_exact2, pk, n_blocks);
  tmem_st_rows16_p8(tP + 48, pk);
  if (kLse) {
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      float sum_a, sum_b;
      unpack_f32x2(sum_exact2[hi], sum_a, sum_b);
      st.l_exact[hi] += sum_a + sum_b;
    }
  }
  tmem_wait_st();
  tc_fence_before();
  if (elect_one()) mbar_arrive(smem_u32(&bars->p_full[me.t][odd]));
  return true;
}

// The row sums move to the column after theirs (see kFlushSteps).  Thread 0 of a quad has both columns, the others zeros.
// last: the tile's latest step; its P V has to be done, and the next one waits for this warp's next P.
__device__ __forceinline__ bool flush_row_sums(const SoftmaxThread& me, int last, Barriers* bars, const AttnArgs& a) {
  if (!wait_bar(&bars->o_done[me.t][last & 1], (last >> 1) & 1, bars, a, 32 + me.t, last)) return false;
  tc_fence_after();
  uint32_t l[4];
  tmem_ld_rows16_c8(me.base + kColL, l);
  tmem_wait_ld();
#pragma unroll
  for (int hi = 0; hi < 2; ++hi) {
    l[2 * hi + 1] = __float_as_uint(__uint_as_float(l[2 * hi]) + __uint_as_float(l[2 * hi + 1]));
    l[2 * hi] = 0u;
  }
  tmem_st_rows16_c8(me.base + kColL, l);
  return true;
}

// What the epilogue of a work item needs of its rows' running state (shared memory; a row's warp writes and reads it).
struct RowResults {
  float neg_m[kQTiles * kTileQ];     // minus the reference maximum
  float l_exact[kQTiles * kTileQ];   // sum of the unrounded exponentials: log-sum-exp output only
};

// 16 rows x 16 dimensions of a 128-byte-swizzled tile of 64 values a row (`row`: shared-memory address of the row that this lane
// points at, 16 h + lane % 16 of the tile's quarter; `chunk`: which 16 bytes of it, 2 k + lane / 16), in the layout of O: register 0:
// block 2 k of 8 dimensions of the thread's first row, 1: of its second row, 2 and 3: block 2 k + 1.
__device__ __forceinline__ uint32_t row_chunk(uint32_t row, int lane, int k) {
  return row + (((2 * k + (lane >> 4)) ^ (lane & 7)) << 4);
}
__device__ __forceinline__ void ld_rows16(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void st_rows16(uint32_t addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3) : "memory");
}

// Epilogue of a work item: diagonal and mean-fill terms, normalisation, store of the warp's 16 rows.  n: the item's number in this
// CTA, last: the tile's latest key step, the item's last.
//
// The queries' own Q, K and V rows and the mean pair are in shared memory (the producer brings them while the item runs).  A thread
// has two rows, and of each block of 8 dimensions the pair 2 i, 2 i + 1, as in O: ldmatrix gives rows of a tile in that layout, and
// stmatrix turns the result into rows, which are stored 128 contiguous bytes at a time.
//
// An item boundary is bound by instructions: all four warps of a scheduler are in it at once.  Before, with the own rows and the mean
// pair read from global memory 16 bytes per thread, V and the result turned around by shuffles within the quad, and the item found
// anew by every warp, a boundary cost the layer 1,215 instructions a warp, as many as 4.6 key steps, and the last epilogue of a launch
// 4,900 clocks.  Layer of 10 frames of 37 x 37, a quarter retained, 280 -> 272.5 us, of 31 frames of 28 x 37, a ninth retained, with
// log-sum-exp 896 -> 874 us, of 4 frames of 16 x 16 17.1 -> 16.7 us, frame attention of 100 frames of 37 x 37 1122 -> 1099 us, of 10 122.5 -> 120.3 us.
template <bool kLse, bool kExtra>
__device__ __forceinline__ bool softmax_epilogue(const AttnArgs& a, Barriers* bars, const SoftmaxThread& me, const RowResults* res,
                                                 const ItemInfo* infos, const SmemLayout& sm, int n, int last) {
  const Plan& pl = a.pl;
  const ItemInfo& info = infos[n % kInfos];
  const int t = me.t, head = info.head, first = info.first[t], end = info.last[t];
  const int i = me.lane & 3;                             // position in the quad
  const int lane0 = 32 * me.q + 16 * me.h;               // the warp's first row within the tile
  const int row0 = info.q0[t] + lane0;                   // ... and in the sequence; the thread's rows: + lane / 4, + lane / 4 + 8
  const uint32_t at = static_cast<uint32_t>(t) * kTileBytes + static_cast<uint32_t>(lane0 + (me.lane & 15)) * (kHeadDim * 2);

  // base-2 logits of the two extra columns (every thread runs the shuffles; rows without the term carry what is not used)
  float l_d[2] = {-INFINITY, -INFINITY}, l_m[2] = {-INFINITY, -INFINITY};
  if (kExtra) {
    bool dropped[2] = {false, false};
    if (a.use_diag) {   // lanes 0..15: a row each
      const int row = row0 + (me.lane & 15);
      bool mine = row >= first && row < end;
      if (mine) mine = a.slot_of_token != nullptr ? a.slot_of_token[row] < 0 : compact_position(a.rule, pl, row) < 0;
      const uint32_t rows = __ballot_sync(kFullMask, mine) >> (me.lane >> 2);
      dropped[0] = (rows & 1) != 0;
      dropped[1] = (rows & 0x100) != 0;
    }
    const uint32_t q_row = smem_u32(sm.q) + (n & 1) * (kQTiles * kTileBytes) + at, k_row = smem_u32(sm.own_k) + at;
    if (!wait_bar(&bars->q_full[n & 1], (n >> 1) & 1, bars, a, 52, n)) return false;
    if (!wait_bar(&bars->own_full, n & 1, bars, a, 53, n)) return false;
    float d[2] = {0.f, 0.f};
    uint64_t m[2] = {pack_f32x2(0.f, 0.f), pack_f32x2(0.f, 0.f)};
#pragma unroll
    for (int k = 0; k < kHeadDim / 16; ++k) {
      uint32_t q[4], own[4];
      ld_rows16(row_chunk(q_row, me.lane, k), q);
      if (a.use_diag) {
        ld_rows16(row_chunk(k_row, me.lane, k), own);
#pragma unroll
        for (int c = 0; c < 4; ++c) d[c & 1] = fma_bf16x2_to_f32(q[c], own[c], d[c & 1]);
      }
      if (a.use_mean) {
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const uint64_t mean = *reinterpret_cast<const uint64_t*>(sm.means + 16 * k + 8 * b + 2 * i);
          m[0] = fma_f32x2(unpack_bf16x2(q[2 * b]), mean, m[0]);
          m[1] = fma_f32x2(unpack_bf16x2(q[2 * b + 1]), mean, m[1]);
        }
      }
    }
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      if (a.use_diag) {
        const float dot = quad_sum(d[hi]);
        if (dropped[hi]) l_d[hi] = dot * a.scale_log2;
      }
      if (a.use_mean) {
        float m0, m1;
        unpack_f32x2(m[hi], m0, m1);
        l_m[hi] = fmaf(quad_sum(m0 + m1), a.scale_log2, a.log2_count[dropped[hi] ? 1 : 0]);
      }
    }
    __syncwarp();
    if (elect_one()) mbar_arrive(smem_u32(&bars->q_empty[n & 1]));
  }

  uint32_t l[4] = {0u, 0u, 0u, 0u};   // thread 0 of a quad: the row sums, in two parts, in registers 0 + 1 (row 0) and 2 + 3 (row 1)
  uint32_t o[2][16];   // register 4 b + 2 hi + e of a half: row hi, output dimension 32 half + 8 b + 2 i + e; zero with no retained keys
#pragma unroll
  for (int half = 0; half < 2; ++half)
#pragma unroll
    for (int c = 0; c < 16; ++c) o[half][c] = 0u;
  if (a.n_kv_tiles > 0) {
    if (!wait_bar(&bars->o_done[t][last & 1], (last >> 1) & 1, bars, a, 50 + t, last)) return false;
    tc_fence_after();
    tmem_ld_rows16_c8(me.base + kColL, l);
    tmem_ld_rows16_c32(me.base + kColO, o[0]);
    tmem_ld_rows16_c32(me.base + kColO + 32, o[1]);
    tmem_wait_ld();
    // O_t has been read: the next work item's first P V may overwrite it
    tc_fence_before();
    if (elect_one()) mbar_arrive(smem_u32(&bars->o_free[t]));
  }
  uint64_t w_s[2], w_d[2], w_m[2];   // weights of the accumulator, of the row's own V and of the mean Value
#pragma unroll
  for (int hi = 0; hi < 2; ++hi) {
    const int r = lane0 + (me.lane >> 2) + 8 * hi;
    // the row's sums: of the rounded probabilities (the normaliser), of the unrounded ones (log-sum-exp)
    const float l_run = __shfl_sync(kFullMask, __uint_as_float(l[2 * hi]) + __uint_as_float(l[2 * hi + 1]), me.lane & ~3);
    float p_d = 0.f, p_m = 0.f, a_s = 1.0f, m_fin = 0.f;
    if (kExtra || kLse) {
      const float m = -res->neg_m[t * kTileQ + r];
      m_fin = m;
      if (kExtra) {
        m_fin = fmaxf(m, fmaxf(l_d[hi], l_m[hi]));
        a_s = exp2f(m - m_fin);
        p_d = exp2f(l_d[hi] - m_fin);              // 0 when the term is absent
        p_m = exp2f(l_m[hi] - m_fin);
      }
    }
    const float z = fmaf(l_run, a_s, p_d + p_m);
    const float inv_z = __fdividef(1.0f, z);   // z is at least one exponential of a row maximum, far from the ends of the range
    w_s[hi] = pack_f32x2(a_s * inv_z, a_s * inv_z);
    w_d[hi] = pack_f32x2(p_d * inv_z, p_d * inv_z);
    w_m[hi] = pack_f32x2(p_m * inv_z, p_m * inv_z);
    if (kLse && i == 0) {
      const int row = info.q0[t] + r;
      const float z_exact = fmaf(res->l_exact[t * kTileQ + r], a_s, p_d + p_m);
      if (row >= first && row < end)
        a.lse[static_cast<size_t>(row) * pl.H + head] = (m_fin + log2f(z_exact)) * 0.6931471805599453f;
    }
  }
  const uint32_t v_row = smem_u32(sm.own_v) + at;
#pragma unroll
  for (int k = 0; k < kHeadDim / 16; ++k) {
    uint32_t own[4], w[4];
    if (kExtra && a.use_diag) ld_rows16(row_chunk(v_row, me.lane, k), own);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int hi = c & 1, reg = 4 * (2 * (k & 1) + (c >> 1)) + 2 * hi;
      uint64_t v = mul_f32x2(pack_f32x2(__uint_as_float(o[k >> 1][reg]), __uint_as_float(o[k >> 1][reg + 1])), w_s[hi]);
      if (kExtra && a.use_diag) v = fma_f32x2(w_d[hi], unpack_bf16x2(own[c]), v);
      if (kExtra && a.use_mean)
        v = fma_f32x2(w_m[hi], *reinterpret_cast<const uint64_t*>(sm.means + kHeadDim + 16 * k + 8 * (c >> 1) + 2 * i), v);
      w[c] = pack_bf16x2(v);
    }
    __syncwarp();   // every lane has its part of V
    st_rows16(row_chunk(v_row, me.lane, k), w[0], w[1], w[2], w[3]);
  }
  __syncwarp();
  // four rows at a time, eight lanes x 16 bytes per row
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int r = 4 * k + (me.lane >> 3), row = row0 + r;
    if (row >= first && row < end) {
      const uint8_t* src = sm.own_v + t * kTileBytes + (lane0 + r) * (kHeadDim * 2) + (((me.lane ^ r) & 7) << 4);
      uint4* dst = reinterpret_cast<uint4*>(a.O + (static_cast<size_t>(row) * pl.H + head) * kHeadDim) + (me.lane & 7);
      *dst = *reinterpret_cast<const uint4*>(src);
    }
  }
  if (kExtra) fence_proxy_async_smem();   // the next copy of own rows comes after these accesses
  __syncwarp();
  if (kExtra && elect_one()) mbar_arrive(smem_u32(&bars->own_empty));
  return true;
}

// The work items of a softmax thread.  The epilogue of an item runs after the first step of the next item: by then its last
// P V has completed, the next item's P V waits for O to be read out (o_free) but its scores do not, and the tensor core and the
// copies are a step ahead.
template <bool kLse, bool kExtra>
__device__ __forceinline__ void softmax_items(const AttnArgs& a, Barriers* bars, const SoftmaxThread& me, RowResults* res, const ItemInfo* infos,
                                              const SmemLayout& sm) {
  const int n_kv = a.n_kv_tiles;
  const int t = me.t;
  const bool ragged = a.last_tile_keys != 0;
  bool res_rows = false;   // the warp had rows in the item before
  int gj = 0;              // this tile's key steps so far, over all work items of the CTA: the phase of the per-step barriers
  bool pending = false;    // the epilogue of the item before
  int n = 0;               // items so far
#pragma unroll 1
  for (uint32_t item = blockIdx.x;; item += gridDim.x, ++n) {
    const bool have = item < static_cast<uint32_t>(a.n_work);
    if (!have && !pending) return;
    RowState st;
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      st.neg_m[hi] = INFINITY;
      st.look_above[hi] = -INFINITY;
      st.l_exact[hi] = 0.f;
    }
    bool active = false, rows = false;   // the tile takes part in this item, the warp has rows in it
    if (have) {
      if (!wait_bar(&bars->info_full[n % kInfos], (n / kInfos) & 1, bars, a, 54, n)) return;
      const ItemInfo& info = infos[n % kInfos];
      active = info.active[t] != 0;
      const int row0 = info.q0[t] + 32 * me.q + 16 * me.h;   // the warp's first row
      rows = row0 + 16 > info.first[t] && row0 < info.last[t];
    }
    int left = active ? n_kv : 0;
    // steps up to the next multiple of kFlushSteps of the item's own, so that a row's sums do not depend on the item's place
    int most = pending ? 1 : kFlushSteps;
#pragma unroll 1
    do {
      const int chunk = left < most ? left : most;
      left -= chunk;
      const int stop = gj + chunk;
      if (rows) {
        // the ragged last tile apart, with every exponential on the special-function unit, where -inf gives an exact 0
        const int full = left == 0 && ragged ? stop - 1 : stop;
#pragma unroll 1
        for (; gj < full; ++gj)
          if (!softmax_step<false, kLse, kPolyBlocks>(me, gj, kTileKV, st, bars, a)) return;
        if (gj < stop) {
          if (!softmax_step<true, kLse, 0>(me, gj, a.last_tile_keys, st, bars, a)) return;
          ++gj;
        }
      } else {   // nothing to compute: the warp's share of S and P is released at once
#pragma unroll 1
        for (; gj < stop; ++gj) {
          if (!wait_bar(&bars->s_full[t], gj & 1, bars, a, 40 + t, gj)) return;
          if (me.lane == 0) {
            mbar_arrive(smem_u32(&bars->s_free[t]));
            mbar_arrive(smem_u32(&bars->p_full[t][gj & 1]));
          }
        }
      }
      if (pending) {
        if (res_rows) {
          if (!softmax_epilogue<kLse, kExtra>(a, bars, me, res, infos, sm, n - 1, stop - chunk - 1)) return;
        } else {
          if (n_kv > 0) {
            // Not before the item's last P V: a warp without rows could otherwise be an item ahead and arrive a second time in
            // the phase in which another warp has not yet read O.
            const int last = stop - chunk - 1;
            if (!wait_bar(&bars->o_done[t][last & 1], (last >> 1) & 1, bars, a, 51, last)) return;
            if (me.lane == 0) mbar_arrive(smem_u32(&bars->o_free[t]));
          }
          if (kExtra) {   // (nor before the item's own rows have come, for the same reason)
            if (!wait_bar(&bars->own_full, (n - 1) & 1, bars, a, 53, n)) return;
            if (me.lane == 0) {
              mbar_arrive(smem_u32(&bars->q_empty[(n - 1) & 1]));
              mbar_arrive(smem_u32(&bars->own_empty));
            }
          }
        }
        pending = false;
        most = kFlushSteps - 1;
      } else {
        if (left > 0 && rows && !flush_row_sums(me, gj - 1, bars, a)) return;
        most = kFlushSteps;
      }
    } while (left > 0);
    if (!have) return;
    pending = active;
    __syncwarp();   // every lane has read the results of the item before, and the record
    if (!active) {
      if (elect_one()) mbar_arrive(smem_u32(&bars->sat_out[n & 1]));
      continue;
    }
#pragma unroll
    for (int hi = 0; hi < 2; ++hi) {
      const int at = t * kTileQ + 32 * me.q + 16 * me.h + (me.lane >> 2) + 8 * hi;
      const float l_exact = kLse ? quad_sum(st.l_exact[hi]) : 0.f;
      if ((me.lane & 3) == 0) {
        res->neg_m[at] = st.neg_m[hi];
        if (kLse) res->l_exact[at] = l_exact;
      }
    }
    __syncwarp();
    res_rows = rows;
  }
}

template <bool kLse, bool kExtra>
__device__ __forceinline__ void softmax_role(const AttnArgs& a, Barriers* bars, RowResults* res, const ItemInfo* infos, const SmemLayout& sm,
                                             uint32_t tmem, int warp, int lane) {
  SoftmaxThread me;
  me.t = warp >> 3;
  me.h = (warp >> 2) & 1;
  me.q = warp & 3;
  me.lane = lane;
  me.base = tmem + me.t * kTmemTileStride + (static_cast<uint32_t>(32 * me.q + 16 * me.h) << 16);   // TMEM lane = row
  softmax_items<kLse, kExtra>(a, bars, me, res, infos, sm);
}

// Value columns 64..79 of a slice of 16 keys, in the 128-byte-swizzled layout of the V tiles: column 64 all ones, the others
// zero, so that P V sums the rows of P on the tensor core.  It is the sum of the bf16-rounded probabilities that the value
// product uses, in fp32, and it costs the softmax warps nothing (adding the rounded values up took one instruction per score
// of the 6.5 that a score took).  128-byte rows: only 32 bytes of each are read.
__device__ __forceinline__ void ones_block(uint8_t* ones, int tid) {
  if (tid < static_cast<int>(kOnesBytes / 16)) {
    const int row = tid >> 3, chunk = tid & 7;
    const uint32_t first = chunk == (row & 7) ? 0x3f80u : 0u;   // bf16 1 in the row's first value
    *reinterpret_cast<uint4*>(ones + tid * 16) = make_uint4(first, 0u, 0u, 0u);
  }
  fence_proxy_async_smem();
}

// kLse: write the log-sum-exp.  kExtra: there is a diagonal or a mean column (frame attention and the dense layer have neither).
template <bool kLse, bool kExtra>
__global__ void __launch_bounds__(kThreads, 1)
global_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_own_k,
                   const __grid_constant__ CUtensorMap tm_own_v, const AttnArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  SmemLayout sm;
  sm.q = smem;
  sm.k = smem + 2 * kQTiles * kTileBytes;
  sm.v = sm.k + kStages * kKeyTileBytes;
  sm.ones = sm.v + kStages * kKeyTileBytes;
  sm.own_v = sm.ones + kOnesBytes;
  sm.own_k = sm.own_v + kQTiles * kTileBytes;
  sm.means = reinterpret_cast<float*>(sm.own_k + kQTiles * kTileBytes);
  __shared__ RowResults row_results;
  __shared__ Barriers bars;
  __shared__ ItemInfo infos[kInfos];

  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);   // warp-uniform by construction
  init_barriers<kExtra>(&bars, a, tid);
  if (warp == kTmemWarp) {
    tmem_alloc(smem_u32(&bars.tmem_base), kTmemCols);
    tmem_relinquish();
  }
  // The first item is found while other warps prepare the rest (found after them, behind a read of the status word and with one thread
  // initialising the barriers, the first key step came 2,000 clocks later: 4 frames of 16 x 16 16.8 -> 15.8 us, one frame of 37 x 37
  // 16.6 -> 15.6 us).
  WorkItem wi = {};
  QueryTile tile0 = {}, tile1 = {};
  if (warp == kTmaWarp) {
    wi = work_item<!kExtra>(a, blockIdx.x);
    tile0 = query_tile(a, wi, 0);
    tile1 = query_tile(a, wi, 1);
    if (elect_one()) {
      prefetch_tensormap(&tm_q);
      prefetch_tensormap(&tm_k);
      prefetch_tensormap(&tm_v);
      if (kExtra) {
        prefetch_tensormap(&tm_own_k);
        prefetch_tensormap(&tm_own_v);
      }
    }
    __syncwarp();
  } else if (warp < kSoftmaxWarps) {
    ones_block(sm.ones, tid);
  }
  // everything above may run while the kernel before this one ends
  grid_dependency_wait();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_base;

  if (warp < kSoftmaxWarps) {
    reg_inc<kRegsSoftmax>();
    softmax_role<kLse, kExtra>(a, &bars, &row_results, infos, sm, tmem, warp, tid & 31);
  } else {
    reg_dec<kRegsOther>();
    if (warp == kTmaWarp) producer_role<!kExtra>(&tm_q, &tm_k, &tm_v, &tm_own_k, &tm_own_v, a, &bars, infos, sm, wi, tile0, tile1);
    else if (warp == kMmaWarp) mma_role<0, !kExtra>(a, &bars, sm, tmem);
    else if (warp == kMmaWarp + 1) mma_role<1, !kExtra>(a, &bars, sm, tmem);
  }

  // a role that left on a wait that ran out may have tensor-memory loads or stores in flight
  tmem_wait_ld();
  tmem_wait_st();
  tc_fence_before();
  __syncthreads();
  if (warp == kTmemWarp) tmem_dealloc(tmem, kTmemCols);
}

// The status block of a launch that no compaction precedes.
__global__ void clear_status_kernel(uint32_t* status) {
  grid_dependency_wait();
  grid_launch_dependents();
  if (threadIdx.x < kAttnStatusBytes / 4) status[threadIdx.x] = 0u;
}

// kExtra: with the query rows' own K and the mean pair
constexpr size_t attn_smem_bytes(bool extra) {
  return static_cast<size_t>(kTileBytes) * (2 * kQTiles) + static_cast<size_t>(kKeyTileBytes) * (2 * kStages) + kOnesBytes +
         kQTiles * kTileBytes + (extra ? kQTiles * kTileBytes + 2 * kHeadDim * sizeof(float) : 0) + 1024;
}

}  // namespace

cudaError_t launch_clear_status(void* status, cudaStream_t st) {
  return launch_dependent(clear_status_kernel, 1, 64, 0, st, static_cast<uint32_t*>(status));
}

size_t global_attn_ws_bytes(const Plan&, int) { return kAttnStatusBytes; }

namespace {

// Once per device: the dynamic shared-memory limit of the kernel, and a check that the launch allocates the
// registers the role split hands out.  setmaxnreg.inc waits, without a time limit, for registers that other
// warps release; if the compiler gave the kernel fewer than kRegsLaunch registers per thread the pool could
// never cover the softmax warps' share and the kernel would hang, so such a build refuses to launch.
typedef void (*AttnKernel)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const AttnArgs);
constexpr AttnKernel kAttnKernels[4] = {global_attn_kernel<false, false>, global_attn_kernel<false, true>,
                                        global_attn_kernel<true, false>, global_attn_kernel<true, true>};

cudaError_t prepare_kernels() {
  static std::mutex mu;
  static bool ready[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (ready[dev]) return cudaSuccess;
  for (int which = 0; which < 4; ++which) {
    const AttnKernel k = kAttnKernels[which];
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, k);
    if (e != cudaSuccess) return e;
    if (fa.numRegs * (kThreads / 32) < kRegsSoftmax * kSoftmaxWarps + kRegsOther * (kThreads / 32 - kSoftmaxWarps))
      return cudaErrorLaunchOutOfResources;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(attn_smem_bytes((which & 1) != 0)));
    if (e != cudaSuccess) return e;
  }
  ready[dev] = true;
  return cudaSuccess;
}

// Query rows of a work item: 256, or, in a launch of one or two rounds of the chip, 160, 144 or 128 where that ends sooner
// by this measure: an item of r <= 160 rows takes 0.68 + 0.32 r / 256 of a full one's time (measured at 128: 0.84; the key steps
// are a chain; between 160 and 256 some scheduler has four warps with work again), and the ragged last items of a kShortLast launch fill up the last round of the others.  2,748 queries x 732 keys
// x 16 heads, 176 items of 256 rows or 288 of 160: 28.5 against 25.6 us; frame attention of two frames of 1,374 tokens 35.8
// against 31.9.  Longer launches keep 256: there the gain is small, and rows that do not exist cost power.
int choose_item_rows(int64_t rows, int64_t problems, int sm_count, bool short_last) {
  const auto rounds = [&](int64_t items) { return (items + sm_count - 1) / sm_count; };
  const auto cost = [](int64_t r) { return 0.68 + 0.32 * static_cast<double>(r) / (kQTiles * kTileQ); };
  const auto end = [&](int r) {
    if (!short_last) return static_cast<double>(rounds((rows + r - 1) / r * problems)) * cost(r);
    const int64_t full = rows / r * problems, last = rows % r != 0 ? problems : 0;
    const int64_t idle = rounds(full) * sm_count - full;
    return static_cast<double>(rounds(full)) * cost(r) + (last > idle ? static_cast<double>(rounds(last - idle)) * cost(rows % r) : 0.0);
  };
  int best = kQTiles * kTileQ;
  if (rounds((rows + best - 1) / best * problems) > 2) return best;
  double least = 0.97 * end(best);   // (not for next to nothing)
  for (int r = 160; r >= kTileQ; r -= 16)
    if (end(r) < least) {
      least = end(r);
      best = r;
    }
  return best;
}

// Frames x heads in a window of frame attention's items (work_item): all, or, where Q, K, V and O are more than L2 holds, as many
// frames as move 32 MB, so that the ragged items find their frame's keys and values still there.  At 30 frames of 1,374 tokens
// and 16 heads one window read 426 MB where Q, K and V are 253; 100 frames 1162 -> 1139 us (windows of 24, 48, 64 and 100 MB
// 1144, 1143, 1147 and 1153; one frame 1146); 10 frames, which fit L2, are no faster.
int32_t choose_window(const Plan& pl) {
  const int64_t mb = int64_t(1) << 20, frame_bytes = 4 * static_cast<int64_t>(pl.L) * pl.H * pl.d * 2;
  if (frame_bytes * pl.n_frames <= 128 * mb) return pl.n_frames * pl.H;
  const int64_t frames = 32 * mb / frame_bytes;
  return static_cast<int32_t>(frames > 1 ? frames : 1) * pl.H;
}

// Tensor maps and launch shared by the two entry points.  frame_mode: see AttnArgs.
cudaError_t launch_attn(const Plan& pl, int sm_count, bool frame_mode, const void* Q, const void* K, const void* V, const void* Kc,
                        const void* Vc, const float* kmean, const float* vmean, void* O, float* lse, void* ws,
                        cudaStream_t st, bool* tmap_failed, const int32_t* slot_of_token, bool status_cleared) {
  *tmap_failed = false;
  AttnArgs a;
  a.pl = pl;
  a.slot_of_token = slot_of_token;
  a.kmean = kmean;
  a.vmean = vmean;
  a.O = static_cast<__nv_bfloat16*>(O);
  a.lse = lse;
  a.status = static_cast<uint32_t*>(ws);
  a.frame_mode = frame_mode ? 1 : 0;
  a.n_keys = frame_mode ? pl.L : pl.M;
  a.n_kv_tiles = static_cast<int32_t>((a.n_keys + kTileKV - 1) / kTileKV);
  a.last_tile_keys = static_cast<int32_t>(a.n_keys % kTileKV);
  for (int dropped = 0; dropped < 2; ++dropped) {   // the mean column stands for every dropped column but the query's own
    const int64_t count = pl.n_dropped - dropped;
    a.log2_count[dropped] = count <= 0 ? -INFINITY : pl.mean_fill == AVGGT_MEAN_FILL ? log2f(static_cast<float>(count)) : 0.0f;
  }
  a.use_diag = (!frame_mode && pl.diag != 0 && pl.n_dropped > 0) ? 1 : 0;
  a.use_mean = (!frame_mode && pl.mean_fill != 0 && pl.n_dropped > 0) ? 1 : 0;
  a.scale_log2 = pl.scale * kLog2e;
  a.inv_scale_log2 = 1.0f / a.scale_log2;
  a.poly_range = (kRescaleThreshold - kLookBelow) * a.inv_scale_log2;
  a.poly_floor = kPolyFloor / a.scale_log2;
  const int64_t rows = frame_mode ? pl.L : pl.n_tok;
  const int64_t problems = static_cast<int64_t>(pl.H) * (frame_mode ? pl.n_frames : 1);
  const bool short_last = !(a.use_diag || a.use_mean);
  a.item_rows = choose_item_rows(rows, problems, sm_count, short_last);
  const int64_t ragged = rows % a.item_rows != 0 ? 1 : 0;
  for (int i = 0; i < 2; ++i) {
    const int n = static_cast<int>(i == 0 || !ragged ? a.item_rows : rows % a.item_rows);
    const int groups = (n + 15) / 16, groups0 = short_last && n <= kTileQ ? groups : (groups + 1) / 2;
    a.split_rows[i] = 16 * groups0;
    a.split_lanes[i] = kTileQ - 16 * (groups - groups0);
  }
  a.pairs = static_cast<int32_t>(rows / a.item_rows + (short_last ? 0 : ragged));
  a.ragged_rows = static_cast<int32_t>(rows % a.item_rows);
  a.by_pairs = make_divisor(a.pairs > 0 ? a.pairs : 1);
  a.by_heads = make_divisor(pl.H);
  a.rule = make_window_rule(pl);
  a.n_problems = static_cast<int32_t>(problems);
  a.window = a.n_problems;
  if (short_last && frame_mode && ragged) a.window = choose_window(pl);
  const int64_t items = a.pairs + (short_last ? ragged : 0);   // of one problem
  a.by_window = make_divisor(static_cast<uint32_t>(a.window * items));
  a.n_work = static_cast<int32_t>(problems * items);

  // token-major [n_tok, H*d] maps for Q and, in frame attention, K and V; head-major [H, M, d] maps for Kc, Vc otherwise
  CUtensorMap tm_q, tm_k, tm_v, tm_own_k, tm_own_v;
  const uint64_t tok_dims[2] = {static_cast<uint64_t>(pl.H) * pl.d, static_cast<uint64_t>(pl.n_tok)};
  const uint64_t tok_str[1] = {static_cast<uint64_t>(pl.H) * pl.d * 2};
  const uint32_t q_box[2] = {kHeadDim, kTileQ};
  bool good = make_tmap_bf16(&tm_q, Q, 2, tok_dims, tok_str, q_box);
  if (frame_mode) {
    const uint32_t kv_box[2] = {kHeadDim, kTileKV};
    good = good && make_tmap_bf16(&tm_k, K, 2, tok_dims, tok_str, kv_box);
    good = good && make_tmap_bf16(&tm_v, V, 2, tok_dims, tok_str, kv_box);
  } else if (pl.M > 0) {
    const uint64_t c_dims[3] = {static_cast<uint64_t>(pl.d), static_cast<uint64_t>(pl.M), static_cast<uint64_t>(pl.H)};
    const uint64_t c_str[2] = {static_cast<uint64_t>(pl.d) * 2, static_cast<uint64_t>(pl.M) * pl.d * 2};
    const uint32_t c_box[3] = {kHeadDim, kTileKV, 1};
    good = good && make_tmap_bf16(&tm_k, Kc, 3, c_dims, c_str, c_box);
    good = good && make_tmap_bf16(&tm_v, Vc, 3, c_dims, c_str, c_box);
  } else {
    tm_k = tm_v = tm_q;   // not read
  }
  if (a.use_diag) {   // the query rows' own K and V
    good = good && make_tmap_bf16(&tm_own_k, K, 2, tok_dims, tok_str, q_box);
    good = good && make_tmap_bf16(&tm_own_v, V, 2, tok_dims, tok_str, q_box);
  } else {
    tm_own_k = tm_own_v = tm_q;   // not read
  }
  if (!good) { *tmap_failed = true; return cudaSuccess; }

  cudaError_t e = prepare_kernels();
  if (e != cudaSuccess) return e;
  if (!status_cleared) {
    e = launch_clear_status(ws, st);
    if (e != cudaSuccess) return e;
  }
  const unsigned grid = static_cast<unsigned>(a.n_work < sm_count ? a.n_work : sm_count);
  const int which = (lse != nullptr ? 2 : 0) + (a.use_diag || a.use_mean ? 1 : 0);
  return launch_dependent(kAttnKernels[which], grid, kThreads, attn_smem_bytes((which & 1) != 0), st, tm_q, tm_k, tm_v, tm_own_k, tm_own_v, a);
}

}  // namespace

cudaError_t launch_global_attn(const Plan& pl, int sm_count, const void* Q, const void* K, const void* V,
                               const void* Kc, const void* Vc, const float* kmean, const float* vmean, void* O,
                               float* lse, void* ws, cudaStream_t st, bool* tmap_failed, const int32_t* slot_of_token,
                               bool status_cleared) {
  return launch_attn(pl, sm_count, false, Q, K, V, Kc, Vc, kmean, vmean, O, lse, ws, st, tmap_failed, slot_of_token,
                     status_cleared);
}

cudaError_t launch_frame_attn(const Plan& pl, int sm_count, const void* Q, const void* K, const void* V, void* O, float* lse,
                              void* ws, cudaStream_t st, bool* tmap_failed) {
  return launch_attn(pl, sm_count, true, Q, K, V, nullptr, nullptr, nullptr, nullptr, O, lse, ws, st, tmap_failed, nullptr, false);
}

}  // namespace avggt
