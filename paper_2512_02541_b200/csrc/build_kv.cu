// K/V compaction and mean-fill reduction (Sec. 4.3 of the AVGGT paper):
// one pass over K and V that copies the retained rows into the head-major
// compact arrays and sums the dropped patch rows for the mean Key/Value pair.
//
// Memory-bound: every row of K and V is read once, retained rows are written once as full 128-byte lines.  Many tokens with a mean:
// build_kv_stream_kernel, contiguous tiles through shared memory; without one (only retained rows are read): build_kv_gather_kernel,
// tiles of compact rows; few tokens: build_kv_small_kernel, a cluster of thread blocks per head.  Sums are kept in
// registers per lane (a lane owns fixed columns), reduced within a block in a fixed order, written as one partial row per block, and
// reduced across blocks by a second small kernel with a fixed shuffle tree: no floating-point
// atomics, so the result does not change from run to run.
#include <mutex>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "tmap.h"

namespace avggt {

namespace {

// The kernels here begin while the kernel before them in the stream, and one before that which has already let it begin, may still
// be writing what they read after their wait: K and V (the projection), the map from tokens to compact positions, a caller's
// list of retained tokens.  They therefore read none of it by the read-only path, which is for data that does not change in a
// kernel's lifetime, or through a pointer the compiler may take for one to such data: K and V by this load, the rest by __ldcg.
__device__ __forceinline__ uint4 ld_stream(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

__device__ __forceinline__ void add_bf16x8(float (&acc)[8], const uint4& v) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    acc[2 * i] += __uint_as_float(w[i] << 16);            // low half: even element
    acc[2 * i + 1] += __uint_as_float(w[i] & 0xffff0000u);  // high half: odd element
  }
}

// Many tokens, with a mean: two thread blocks per SM walk over tiles of consecutive tokens, whose rows of K and V
// (contiguous: two bulk copies) go through a ring of shared-memory stages.  One warp issues the copies and, as a tile arrives, one
// TMA store per retained row and array, which takes the row's heads to their places in the head-major array; the other eight
// warps only add: a thread owns 16 bytes of a row (eight columns) and takes every row of the tile that is dropped.
//
// What bounds it is HBM.  457,542 tokens of 16 heads, a quarter retained (2.37 GB): 396 -> 356 us (6.0 -> 6.7 TB/s) against a warp per
// row with 16 bytes per lane in flight, whose loads stop while it adds and stores; 13,740 tokens 13.9 -> 11.4 us, 137,400
// tokens, a ninth retained, 107.0 -> 102.5.  Stages of 16 + 16 KB, three in each of two blocks per SM: six in one block 377 us (14.0 at 13,740 tokens),
// four 356 (14.3), three of 32 + 32 KB 353 (14.2); of 8 + 8 KB 536 and more in one block (the copying warp's chain of waits per tile),
// 362 in two; two of 16 + 16 KB in two blocks 395, in three 355.
//
// Where a block has a few tiles only, what follows the last copy counts: an adding thread reads four rows before it adds the first of them.
// Row by row, a ninth retained, the kernel was slower than a warp per row: 8,244 tokens of 12 heads 11.8 us against 11.1, now 10.2;
// 5,496 of 20 heads 12.2 against 11.9, now 11.1; 8,244 of 32 heads 18.9 against 18.6, now 18.5; 137,400 of 16 heads 102.5, now 100.2.
constexpr int kStreamSums = 256;                    // adding threads
constexpr int kStreamThreads = kStreamSums + 32;    // and the warp that copies
constexpr int kStreamBlocks = 2;                    // per SM
constexpr int kStreamStages = 3;
constexpr uint32_t kStreamBytes = 16 * 1024;        // of K, and of V, in a stage (at most)
constexpr int kStreamRows = 32;                     // rows of a tile (at most): the copying warp has a lane for each
constexpr int kStreamTogether = 4;                  // rows that an adding thread reads before it adds the first
constexpr int kStreamFlush = 8;                     // tiles after which a thread's sums move on: short chains round less
constexpr size_t kStreamSmemBytes = 2 * kStreamStages * kStreamBytes + 128;

struct StreamArgs {
  Plan pl;
  WindowRule rule;
  const uint8_t* K;
  const uint8_t* V;
  uint4* Kc;           // for rows that a wait which ran out kept from being copied (as kc_rows)
  uint4* Vc;
  int64_t kc_rows;
  int32_t rows;        // of a tile
  int32_t* idx;
  const int32_t* slot_of_token;
  float* partials;     // [gridDim.x][2 * H * d]
  uint32_t* status;
};

struct __align__(8) StreamBarriers {
  uint64_t full[kStreamStages], empty[kStreamStages];
};

// A wait for a copy or for the other warps; false after the time limit.
__device__ __forceinline__ bool stream_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t b = smem_u32(bar);
  if (mbar_try_wait(b, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(b, parity))
    if (globaltimer_ns() - t0 > AVGGT_WAIT_LIMIT_NS) return false;
  return true;
}

// A wait that ran out: in the status block, where the call has one (the attention that follows then does nothing).
__device__ __forceinline__ void stream_report(uint32_t* status, int lane) {
  if (status == nullptr || lane != 0 || atomicCAS(status, 0u, 1u) != 0u) return;
  status[1] = blockIdx.x;
  status[2] = 90;
  status[3] = 0;
}

// Row m of the compact arrays, all heads, by a warp that could not copy it because a wait ran out: NaN, so that a call without a status
// block does not pass for a good one.
__device__ __forceinline__ void mark_row(uint4* Kc, uint4* Vc, int64_t kc_rows, int H, int m, int lane) {
  const uint4 nan = make_uint4(0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu, 0x7fff7fffu);
  for (int c = lane; c < H * 8; c += 32) {
    const size_t at = (static_cast<size_t>(c >> 3) * static_cast<size_t>(kc_rows) + static_cast<size_t>(m)) * 8u + (c & 7);
    Kc[at] = nan;
    Vc[at] = nan;
  }
}

// Build for the wait-limit test only (never part of libavggt.so): in calls of fewer tokens than this the first thread block leaves out the
// copies of its second tile.
#ifdef AVGGT_TEST_SKIP_TILE_LOAD_BELOW
#define AVGGT_SKIP_TILE(n_tok, stage) (blockIdx.x == 0 && (stage) == 1 && (n_tok) < AVGGT_TEST_SKIP_TILE_LOAD_BELOW)
#else
#define AVGGT_SKIP_TILE(n_tok, stage) false
#endif

// PASSES: chunks of 16 bytes per adding thread (2 * H * 8 of them in a row of K and V).
template <int PASSES>
__global__ void __launch_bounds__(kStreamThreads, kStreamBlocks)
build_kv_stream_kernel(const __grid_constant__ CUtensorMap tm_kc, const __grid_constant__ CUtensorMap tm_vc, const StreamArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  __shared__ StreamBarriers bars;
  __shared__ uint32_t kept_mask[kStreamStages];
  __shared__ float red[PASSES == 1 ? kStreamSums * 8 : 1];
  const Plan& pl = a.pl;
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const uint32_t row_bytes = static_cast<uint32_t>(pl.H) * 128u, n_tok = static_cast<uint32_t>(pl.n_tok);
  const uint32_t rows = a.rows, n_tiles = (n_tok + rows - 1) / rows;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStreamStages; ++s) {
      mbar_init(smem_u32(&bars.full[s]), 2);
      mbar_init(smem_u32(&bars.empty[s]), kStreamSums / 32);
    }
    fence_mbar_init();
  }
  grid_dependency_wait();
  if (blockIdx.x == 0 && a.status != nullptr && threadIdx.x < kAttnStatusBytes / 4) a.status[threadIdx.x] = 0u;
  __syncthreads();

  if (warp == kStreamSums / 32) {
    if (lane == 0 && pl.M > 0) {
      prefetch_tensormap(&tm_kc);
      prefetch_tensormap(&tm_vc);
    }
    // compact position of the row of tile t that this lane stands for, -1 if it is dropped, -2 if it does not exist
    const auto position = [&](uint32_t t) {
      const uint32_t row = t * rows + lane;
      if (t >= n_tiles || lane >= static_cast<int>(rows) || row >= n_tok) return -2;
      return a.slot_of_token != nullptr ? __ldcg(a.slot_of_token + row) : compact_position(a.rule, pl, row);
    };
    const auto load = [&](uint32_t t, int stage) {
      if (lane == 0 && !AVGGT_SKIP_TILE(n_tok, stage)) {
        const uint32_t row0 = t * rows, n = n_tok - row0 < rows ? n_tok - row0 : rows;
        const uint32_t fb = smem_u32(&bars.full[stage]), dst = smem_u32(stages + 2 * stage * kStreamBytes);
        mbar_arrive_expect_tx(fb, 2 * n * row_bytes);
        bulk_load(dst, a.K + static_cast<size_t>(row0) * row_bytes, n * row_bytes, fb);
        bulk_load(dst + kStreamBytes, a.V + static_cast<size_t>(row0) * row_bytes, n * row_bytes, fb);
      }
    };
    const auto tell = [&](int stage, int m) {   // the adding warps which rows of the tile are retained; m: the lane's position
      const uint32_t mask = __ballot_sync(0xffffffffu, m >= 0);
      if (lane == 0) {
        kept_mask[stage] = mask;
        mbar_arrive(smem_u32(&bars.full[stage]));
      }
      __syncwarp();
    };
    int pos[kStreamStages];   // of the lane's row, by stage
#pragma unroll
    for (int s = 0; s < kStreamStages; ++s) {
      if (blockIdx.x + s * gridDim.x < n_tiles) load(blockIdx.x + s * gridDim.x, s);
    }
#pragma unroll
    for (int s = 0; s < kStreamStages; ++s) {   // under the copies
      pos[s] = position(blockIdx.x + s * gridDim.x);
      if (blockIdx.x + s * gridDim.x < n_tiles) tell(s, pos[s]);
    }
    bool ok = true;
    uint32_t left = n_tiles;   // first tile whose rows are not stored, where a wait ran out
    int round = 0;
    for (uint32_t t0 = blockIdx.x; t0 < n_tiles && ok; t0 += kStreamStages * gridDim.x, ++round) {
#pragma unroll
      for (int s = 0; s < kStreamStages; ++s) {
        const uint32_t t = t0 + s * gridDim.x;
        if (t >= n_tiles || !ok) break;
        const uint32_t refill = t + (kStreamStages - 1) * gridDim.x;   // the tile for the stage before this one
        const int before = s == 0 ? kStreamStages - 1 : s - 1;
        const bool more = refill < n_tiles && (round > 0 || s > 0);
        const int next = more ? position(refill) : -2;
        ok = __all_sync(0xffffffffu, stream_wait(&bars.full[s], round & 1));
        if (!ok) {
          left = t;
          break;
        }
        const int m = pos[s];
        uint32_t mask = __ballot_sync(0xffffffffu, m >= 0);
        if (m >= 0 && a.idx != nullptr) a.idx[m] = static_cast<int32_t>(t * rows + lane);
        const uint32_t src = smem_u32(stages + 2 * s * kStreamBytes);
        while (mask != 0) {
          const int r = __ffs(mask) - 1;
          mask &= mask - 1;
          const int at = __shfl_sync(0xffffffffu, m, r);
          if (lane == 0) {
            tma_store_3d(&tm_kc, src + r * row_bytes, 0, 0, at);
            tma_store_3d(&tm_vc, src + kStreamBytes + r * row_bytes, 0, 0, at);
          }
        }
        if (lane == 0) {
          bulk_commit();
          if (more) bulk_wait_read<1>();   // the stores of the tile before this one have read their stage
        }
        __syncwarp();
        if (more) {
          ok = __all_sync(0xffffffffu, stream_wait(&bars.empty[before], (s == 0 ? round - 1 : round) & 1));
          if (!ok) {
            left = t + gridDim.x;
            break;
          }
          load(refill, before);
          tell(before, next);
          pos[before] = next;
        }
      }
    }
    if (!ok) {   // a wait ran out: whatever is still on its way arrives before the block gives up its shared memory
      stream_report(a.status, lane);
      for (int s = 0; s < kStreamStages; ++s) (void)stream_wait(&bars.full[s], 0), (void)stream_wait(&bars.full[s], 1);
      for (uint32_t t = left; t < n_tiles; t += gridDim.x) {
        const int m = position(t);
        for (uint32_t mask = __ballot_sync(0xffffffffu, m >= 0); mask != 0; mask &= mask - 1)
          mark_row(a.Kc, a.Vc, a.kc_rows, pl.H, __shfl_sync(0xffffffffu, m, __ffs(mask) - 1), lane);
      }
    }
    if (lane == 0) bulk_wait_read<0>();   // the stores complete before the kernel does
    __syncwarp();
  } else {
    const int chunks = pl.H * 16, groups = PASSES == 1 ? kStreamSums / chunks : 1;
    const int group = PASSES == 1 ? static_cast<int>(threadIdx.x) / chunks : 0;
    const int c0 = PASSES == 1 ? static_cast<int>(threadIdx.x) - group * chunks : static_cast<int>(threadIdx.x);
    const int half = pl.H * 8;
    uint64_t run[PASSES][4], sum[PASSES][4];
    uint32_t at[PASSES];
#pragma unroll
    for (int p = 0; p < PASSES; ++p) {
      const int c = c0 + p * kStreamSums;
      at[p] = c < half ? c * 16 : kStreamBytes + (c - half) * 16;
#pragma unroll
      for (int e = 0; e < 4; ++e) run[p][e] = sum[p][e] = pack_f32x2(0.f, 0.f);
    }
    bool ok = true;
    int stage = 0, since = 0;
    uint32_t parity = 0;
    for (uint32_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
      ok = __all_sync(0xffffffffu, stream_wait(&bars.full[stage], parity));
      if (!ok) break;
      const uint8_t* src = stages + 2 * stage * kStreamBytes;
      const uint32_t n = n_tok - t * rows < rows ? n_tok - t * rows : rows;
      const uint32_t kept = kept_mask[stage];
      if (group < groups) {
        for (uint32_t r0 = group; r0 < n; r0 += kStreamTogether * groups) {
          uint4 v[kStreamTogether][PASSES];   // zeros, which add nothing, for a row that is retained or does not exist
#pragma unroll
          for (int i = 0; i < kStreamTogether; ++i) {
            const uint32_t r = r0 + i * groups;
            const bool add = r < n && ((kept >> r) & 1u) == 0;
#pragma unroll
            for (int p = 0; p < PASSES; ++p) {
              v[i][p] = make_uint4(0u, 0u, 0u, 0u);
              if (add && (PASSES == 1 || c0 + p * kStreamSums < chunks)) v[i][p] = *reinterpret_cast<const uint4*>(src + at[p] + r * row_bytes);
            }
          }
#pragma unroll
          for (int i = 0; i < kStreamTogether; ++i)
#pragma unroll
            for (int p = 0; p < PASSES; ++p) {
              run[p][0] = add_f32x2(run[p][0], unpack_bf16x2(v[i][p].x));
              run[p][1] = add_f32x2(run[p][1], unpack_bf16x2(v[i][p].y));
              run[p][2] = add_f32x2(run[p][2], unpack_bf16x2(v[i][p].z));
              run[p][3] = add_f32x2(run[p][3], unpack_bf16x2(v[i][p].w));
            }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars.empty[stage]));
      if (++stage == kStreamStages) { stage = 0; parity ^= 1; }
      if (++since == kStreamFlush) {
        since = 0;
#pragma unroll
        for (int p = 0; p < PASSES; ++p)
#pragma unroll
          for (int e = 0; e < 4; ++e) { sum[p][e] = add_f32x2(sum[p][e], run[p][e]); run[p][e] = pack_f32x2(0.f, 0.f); }
      }
    }
    float* out = a.partials + static_cast<size_t>(blockIdx.x) * (static_cast<size_t>(chunks) * 8);
#pragma unroll
    for (int p = 0; p < PASSES; ++p) {
      const int c = c0 + p * kStreamSums;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float lo, hi;
        unpack_f32x2(add_f32x2(sum[p][e], run[p][e]), lo, hi);
        if (!ok) lo = hi = __int_as_float(0x7fffffff);   // a copy that never came shows in the means
        if (PASSES > 1 || groups == 1) {
          if (group < groups && c < chunks) *reinterpret_cast<float2*>(out + c * 8 + 2 * e) = make_float2(lo, hi);
        } else if (group < groups) {
          red[(group * chunks + c) * 8 + 2 * e] = lo;
          red[(group * chunks + c) * 8 + 2 * e + 1] = hi;
        }
      }
    }
  }
  grid_launch_dependents();
  __syncthreads();
  const int cols = pl.H * 128, groups = kStreamSums / (pl.H * 16);
  if (PASSES == 1 && groups > 1) {   // the groups' sums, in order
    for (int col = threadIdx.x; col < cols; col += kStreamThreads) {
      float s = 0.f;
      for (int g = 0; g < groups; ++g) s += red[g * cols + col];
      a.partials[static_cast<size_t>(blockIdx.x) * cols + col] = s;
    }
  }
}

// Many tokens, nothing to average: only the retained rows are read.  A block is one warp, which walks over tiles of consecutive compact
// rows: a bulk copy per row and array (one per array where the tile's tokens are consecutive) into a stage, and a TMA store of the
// whole tile per array to the head-major places.  HBM is the bound.  Against a warp per token with 16-byte loads: 457,542 tokens of
// 16 heads, a quarter retained (1.0 GB) 233 -> 171 us (5.8 TB/s), 137,400 tokens all retained 203 -> 185 us (6.1 TB/s), 82,440 tokens, a
// ninth retained, 21 -> 10 us, 137,400 tokens of 6 heads, a quarter retained, 38 -> 17 us.
//
// Above 16 heads a block per SM has the three stages, 20 + 20 KB each: with two blocks of 16 + 16 KB a tile is few rows, and where all rows are
// retained the kernel was slower than a warp per token.  A warp per token, two blocks, one of 32 + 32, of 24 + 24 and of 20 + 20 KB, us: 137,400
// tokens of 24 heads 296, 311, 300, 289, 274; of 28 346, 354, 352, 332, 320; 54,960 of 32 160, 165, 161, 160, 157; 137,400 of 20 heads, a quarter
// retained, 109, 70, 68, 67, 65.
constexpr uint32_t kGatherBytesManyHeads = 20 * 1024;
constexpr size_t gather_smem_bytes(uint32_t stage_bytes) { return 2 * kStreamStages * stage_bytes + 128; }
struct GatherArgs {
  Plan pl;
  Divisor by_Lc, by_kept_w;
  const uint8_t* K;
  const uint8_t* V;
  uint4* Kc;           // where a tile is not stored whole (and as in StreamArgs)
  uint4* Vc;
  int64_t kc_rows;
  uint32_t stage_bytes;   // of K, and of V, in a stage
  int32_t rows;        // of a tile
  int32_t* idx;
  const int32_t* caller_idx;   // caller-chosen retained set: token of every compact row; else null
  const int32_t* slot_of_token;   // and compact row of every token: of a token listed twice only this row is written
  uint32_t* status;
  float* zero_kmean;   // mean pair of a problem that drops nothing, or null
  float* zero_vmean;
};

// Token of compact row m by the window rule.
__device__ __forceinline__ int32_t token_of_compact(const GatherArgs& a, uint32_t m) {
  const Plan& pl = a.pl;
  uint32_t f = 0, c = m;
  if (!pl.keep_first) {
    f = divide(m, a.by_Lc, c);
  } else if (m >= static_cast<uint32_t>(pl.L)) {
    f = 1 + divide(m - static_cast<uint32_t>(pl.L), a.by_Lc, c);
  } else {
    return static_cast<int32_t>(m);
  }
  const uint32_t n_special = static_cast<uint32_t>(pl.n_special);
  uint32_t u = c;
  if (c >= n_special) {
    uint32_t col;
    const uint32_t r = divide(c - n_special, a.by_kept_w, col);
    u = n_special + r * pl.s_h * pl.grid_w + col * pl.s_w;
  }
  return static_cast<int32_t>(f * pl.L + u);
}

__global__ void __launch_bounds__(32)
build_kv_gather_kernel(const __grid_constant__ CUtensorMap tm_kc, const __grid_constant__ CUtensorMap tm_vc, const GatherArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  __shared__ __align__(8) uint64_t full[kStreamStages];
  const Plan& pl = a.pl;
  const int lane = threadIdx.x;
  const uint32_t row_bytes = static_cast<uint32_t>(pl.H) * 128u, rows = a.rows, M = static_cast<uint32_t>(pl.M);
  const uint32_t n_tiles = (M + rows - 1) / rows;
  if (lane == 0) {
    for (int s = 0; s < kStreamStages; ++s) mbar_init(smem_u32(&full[s]), 1);
    fence_mbar_init();
    if (M > 0) {
      prefetch_tensormap(&tm_kc);
      prefetch_tensormap(&tm_vc);
    }
  }
  __syncwarp();
  grid_dependency_wait();
  if (blockIdx.x == 0) {
    // what would otherwise be launches of their own: the status block of the attention that follows, and the mean pair of
    // a problem that drops nothing
    if (a.status != nullptr)
      for (int i = lane; i < static_cast<int>(kAttnStatusBytes / 4); i += 32) a.status[i] = 0u;
    if (a.zero_kmean != nullptr)
      for (int i = lane; i < pl.H * pl.d; i += 32) { a.zero_kmean[i] = 0.f; a.zero_vmean[i] = 0.f; }
  }
  // token of the lane's row of tile t; -1 if there is none
  const auto token = [&](uint32_t t) {
    const uint32_t m = t * rows + lane;
    if (t >= n_tiles || lane >= static_cast<int>(rows) || m >= M) return -1;
    if (a.caller_idx == nullptr) return token_of_compact(a, m);
    const int32_t tok = __ldcg(a.caller_idx + m);
    // (entries of a caller's list that are no token are passed over)
    return tok >= 0 && tok < pl.n_tok && __ldcg(a.slot_of_token + tok) == static_cast<int32_t>(m) ? tok : -1;
  };
  const auto load = [&](int stage, int tok) {
    if (AVGGT_SKIP_TILE(pl.n_tok, stage)) return;
    const uint32_t have = __ballot_sync(0xffffffffu, tok >= 0);
    const int tok0 = __shfl_sync(0xffffffffu, tok, 0);
    const uint32_t fb = smem_u32(&full[stage]), dst = smem_u32(stages + 2 * stage * a.stage_bytes);
    const uint32_t bytes = __popc(have) * row_bytes;
    if (lane == 0) mbar_arrive_expect_tx(fb, 2 * bytes);
    __syncwarp();
    // consecutive tokens, from the first row on
    if ((have & (have + 1)) == 0 && __all_sync(0xffffffffu, tok < 0 || tok == tok0 + lane)) {
      if (lane == 0 && have != 0) {
        bulk_load(dst, a.K + static_cast<size_t>(tok0) * row_bytes, bytes, fb);
        bulk_load(dst + a.stage_bytes, a.V + static_cast<size_t>(tok0) * row_bytes, bytes, fb);
      }
    } else if (tok >= 0) {
      bulk_load(dst + lane * row_bytes, a.K + static_cast<size_t>(tok) * row_bytes, row_bytes, fb);
      bulk_load(dst + a.stage_bytes + lane * row_bytes, a.V + static_cast<size_t>(tok) * row_bytes, row_bytes, fb);
    }
    __syncwarp();
  };
  int toks[kStreamStages];   // of the lane's row, by stage
#pragma unroll
  for (int s = 0; s < kStreamStages; ++s) {
    const uint32_t t = blockIdx.x + s * gridDim.x;
    toks[s] = token(t);
    if (t < n_tiles) load(s, toks[s]);
  }
  bool ok = true;
  uint32_t left = n_tiles;   // first tile whose rows are not stored, where a wait ran out
  int round = 0;
  for (uint32_t t0 = blockIdx.x; t0 < n_tiles && ok; t0 += kStreamStages * gridDim.x, ++round) {
#pragma unroll
    for (int s = 0; s < kStreamStages; ++s) {
      const uint32_t t = t0 + s * gridDim.x;
      if (t >= n_tiles) break;
      const uint32_t refill = t + (kStreamStages - 1) * gridDim.x;   // the tile for the stage before this one
      const int before = s == 0 ? kStreamStages - 1 : s - 1;
      const bool more = refill < n_tiles && (round > 0 || s > 0);
      const int next = more ? token(refill) : -1;
      ok = __all_sync(0xffffffffu, stream_wait(&full[s], round & 1));
      if (!ok) {
        left = t;
        break;
      }
      const int tok = toks[s];
      const uint32_t m0 = t * rows;
      if (tok >= 0 && a.idx != nullptr) a.idx[m0 + lane] = tok;
      const uint8_t* src = stages + 2 * s * a.stage_bytes;
      const uint32_t have = __ballot_sync(0xffffffffu, tok >= 0), exist = M - m0 < rows ? M - m0 : rows;
      if (__popc(have) == static_cast<int>(exist)) {
        if (lane == 0) {   // (rows of the box beyond the last compact row are not written: the tensor map ends there)
          tma_store_3d(&tm_kc, smem_u32(src), 0, 0, m0);
          tma_store_3d(&tm_vc, smem_u32(src) + a.stage_bytes, 0, 0, m0);
        }
      } else {   // with rows passed over
        for (uint32_t left_rows = have; left_rows != 0; left_rows &= left_rows - 1) {
          const int r = __ffs(left_rows) - 1;
          for (int c = lane; c < pl.H * 8; c += 32) {
            const size_t at = (static_cast<size_t>(c >> 3) * static_cast<size_t>(a.kc_rows) + m0 + r) * 8u + (c & 7);
            a.Kc[at] = *reinterpret_cast<const uint4*>(src + r * row_bytes + c * 16);
            a.Vc[at] = *reinterpret_cast<const uint4*>(src + a.stage_bytes + r * row_bytes + c * 16);
          }
        }
      }
      if (lane == 0) {
        bulk_commit();
        if (more) bulk_wait_read<1>();   // the stores of the tile before this one have read their stage
      }
      __syncwarp();
      if (more) {
        load(before, next);
        toks[before] = next;
      }
    }
  }
  if (!ok) {   // a wait ran out: whatever is still on its way arrives before the block gives up its shared memory
    stream_report(a.status, lane);
    for (int s = 0; s < kStreamStages; ++s) (void)stream_wait(&full[s], 0), (void)stream_wait(&full[s], 1);
    for (uint32_t t = left; t < n_tiles; t += gridDim.x) {
      for (uint32_t have = __ballot_sync(0xffffffffu, token(t) >= 0); have != 0; have &= have - 1)
        mark_row(a.Kc, a.Vc, a.kc_rows, pl.H, static_cast<int>(t * rows) + __ffs(have) - 1, lane);
    }
  }
  if (lane == 0) bulk_wait_read<0>();   // the stores complete before the kernel does
  __syncwarp();
  grid_launch_dependents();
}

// The same for few tokens, in one launch: a cluster of thread blocks takes one head of K or of V, each block every
// cluster-size-th group of 128 rows, and the blocks put their sums into the first one's shared memory, which adds them up: one barrier
// of the cluster between the last load and the end (with the first block reading from the others there were two, the second so that
// they would stay: layer of 4 frames of 16 x 16 15.8 -> 15.0 us, of one frame of 37 x 37 15.5 -> 14.9 us).  No partial sums in
// global memory (for a few frames as many bytes as K and V themselves) and no second kernel.  A row's 128 bytes of the
// head are read by 8 threads, 16 bytes each, four rows in flight per thread.
constexpr int kSmallThreads = 1024;
constexpr int kSmallRows = kSmallThreads / 8;   // rows a block reads at once

// Up to so many tokens per block of a cluster.  Above, the bytes are the bound.  Times in us, this kernel first, then
// build_kv_stream_kernel with its reduction (148 SMs): 16 heads, clusters of 4, limit 4,400: 4.5 and 5.4 at 1,374 tokens, 7.0 and 7.0 at
// 4,122, 8.1 and 7.5 at 5,496, 15.3 and 9.8 at 10,992.  6 heads, clusters of 8, limit 8,800: 4.2 and 5.1 at 1,374, 6.0 and 6.0 at 5,496,
// 7.1 and 7.5 at 8,244, 8.2 and 7.7 at 10,992.  24 heads, clusters of 2, limit 2,200: 5.8 and 6.0 at 1,374, 8.1 and 7.0 at 2,748.
constexpr int64_t kSmallTokensPerBlock = 1100;

struct SmallArgs {
  Plan pl;
  WindowRule rule;
  const uint4* K;
  const uint4* V;
  uint4* Kc;
  uint4* Vc;
  int64_t kc_rows;
  int32_t* idx;
  const int32_t* slot_of_token;
  float* kmean;        // null: no mean pair
  float* vmean;
  float scale;         // 1 / number of dropped rows, or 1 for the sums; 0: zero-fill
  uint32_t* status;
};

__global__ void __launch_bounds__(kSmallThreads)
build_kv_small_kernel(const SmallArgs a) {
  __shared__ float red[kSmallThreads / 32][64];
  __shared__ float part[8][64];   // in the cluster's first block: the sums of all
  const Plan& pl = a.pl;
  const uint32_t rank = cluster_cta_rank(), n_ranks = cluster_size();
  const int which_head = blockIdx.x / n_ranks;
  const int which = which_head >= pl.H ? 1 : 0, head = which_head - which * pl.H;
  const uint32_t c = threadIdx.x & 7u;
  const uint4* src = (which == 0 ? a.K : a.V) + head * 8 + c;
  uint4* dst = (which == 0 ? a.Kc : a.Vc) + static_cast<size_t>(head) * static_cast<size_t>(a.kc_rows) * 8u + c;
  const uint32_t chunks_per_row = static_cast<uint32_t>(pl.H) * 8u, n_tok = static_cast<uint32_t>(pl.n_tok);
  const bool add = a.kmean != nullptr && a.scale != 0.f;
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;

  if (a.kmean != nullptr) cluster_arrive();
  grid_dependency_wait();
  if (blockIdx.x == 0 && a.status != nullptr && threadIdx.x < kAttnStatusBytes / 4) a.status[threadIdx.x] = 0u;
  constexpr int kInFlight = 4;
  for (uint32_t row0 = rank * kSmallRows + (threadIdx.x >> 3); row0 < n_tok; row0 += kInFlight * n_ranks * kSmallRows) {
    uint4 v[kInFlight];
    int32_t m[kInFlight];
#pragma unroll
    for (int i = 0; i < kInFlight; ++i) {
      const uint32_t row = row0 + i * n_ranks * kSmallRows;
      v[i] = make_uint4(0u, 0u, 0u, 0u);   // beyond the last row: adds nothing
      m[i] = -1;
      if (row < n_tok) {
        m[i] = a.slot_of_token != nullptr ? __ldcg(a.slot_of_token + row) : compact_position(a.rule, pl, row);
        if (m[i] >= 0 || add) v[i] = ld_stream(src + static_cast<size_t>(row) * chunks_per_row);
      }
    }
#pragma unroll
    for (int i = 0; i < kInFlight; ++i) {
      if (m[i] >= 0) {
        dst[static_cast<size_t>(m[i]) * 8u] = v[i];
        if (which_head == 0 && c == 0 && a.idx != nullptr) a.idx[m[i]] = static_cast<int32_t>(row0 + i * n_ranks * kSmallRows);
      } else {
        add_bf16x8(acc, v[i]);
      }
    }
  }
  grid_launch_dependents();
  if (a.kmean == nullptr) return;   // the same for every block of the launch
  // the warp's four rows, then the block's 32 warps, then the cluster's blocks, in a fixed order
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 8);
    acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], 16);
    if ((threadIdx.x & 31) < 8) red[threadIdx.x >> 5][8 * c + e] = acc[e];
  }
  __syncthreads();
  float sum = 0.f;
  if (threadIdx.x < 64) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kSmallThreads / 32; ++w) s += red[w][threadIdx.x];
    sum = s;
  }
  cluster_wait();   // the first block has begun, so that its shared memory can be written
  if (threadIdx.x < 64) st_cluster_f32(cluster_addr(smem_u32(&part[rank][threadIdx.x]), 0), sum);
  cluster_sync();
  if (rank == 0 && threadIdx.x < 64) {
    float s = 0.f;
    for (uint32_t r = 0; r < n_ranks; ++r) s += part[r][threadIdx.x];
    (which == 0 ? a.kmean : a.vmean)[head * 64 + threadIdx.x] = s * a.scale;
  }
}

// out[col] = (sum over blocks of partials[b][col]) / n_dropped, col in [0, 2*cols)
// block = 32 columns x 32 block-groups; the cross-group sum is a warp shuffle tree.
__global__ void __launch_bounds__(1024)
mean_finalize_kernel(const float* partials, int n_blocks, int cols2, float inv_count,
                     float* __restrict__ kmean, float* __restrict__ vmean) {
  __shared__ float tile[32][33];
  grid_launch_dependents();
  grid_dependency_wait();
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int col = blockIdx.x * 32 + c;
  float s = 0.f;
  if (col < cols2) {
    constexpr int kAhead = 10;   // 296 blocks in one go: the loads wait for one another otherwise
    for (int b0 = g; b0 < n_blocks; b0 += 32 * kAhead) {
      float part[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i)
        part[i] = b0 + 32 * i < n_blocks ? __ldcg(partials + static_cast<size_t>(b0 + 32 * i) * cols2 + col) : 0.f;
#pragma unroll
      for (int i = 0; i < kAhead; ++i) s += part[i];
    }
  }
  tile[c][g] = s;
  __syncthreads();
  // warp g now owns column blockIdx.x*32 + g; lane c holds the partial of group c
  float v = tile[g][c];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int ocol = blockIdx.x * 32 + g;
  if (c == 0 && ocol < cols2) {
    const int cols = cols2 / 2;
    if (ocol < cols) kmean[ocol] = v * inv_count;
    else vmean[ocol - cols] = v * inv_count;
  }
}

// slot_of_token[t] = -1 for every token, then m for the m-th retained token.  Entries of idx outside
// [0, n_tok) are skipped.
__global__ void fill_slots_kernel(int32_t* __restrict__ slot_of_token, int64_t n_tok) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n_tok) slot_of_token[i] = -1;
}
__global__ void scatter_slots_kernel(const int32_t* idx, int64_t M, int32_t* __restrict__ slot_of_token, int64_t n_tok) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int64_t m = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (m < M) {
    const int32_t t = __ldcg(idx + m);
    if (t >= 0 && t < n_tok) slot_of_token[t] = static_cast<int32_t>(m);
  }
}

int stream_rows(const Plan& pl, uint32_t stage_bytes = kStreamBytes) {
  const int rows = static_cast<int>(stage_bytes) / (pl.H * 128);
  return rows < kStreamRows ? rows : kStreamRows;
}

// Once per device: the dynamic shared-memory limit.
cudaError_t prepare_stream_kernels() {
  static std::mutex mu;
  static bool ready[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (ready[dev]) return cudaSuccess;
  for (const void* kernel : {reinterpret_cast<const void*>(build_kv_stream_kernel<1>), reinterpret_cast<const void*>(build_kv_stream_kernel<2>)}) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kStreamSmemBytes));
    if (e != cudaSuccess) return e;
  }
  e = cudaFuncSetAttribute(build_kv_gather_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(gather_smem_bytes(kGatherBytesManyHeads)));
  if (e != cudaSuccess) return e;
  ready[dev] = true;
  return cudaSuccess;
}

// The compact arrays as [M, H, d], a head every kc_rows rows: a box is all heads of `rows` rows.
bool make_compact_tmap(CUtensorMap* tm, const Plan& pl, void* base, int64_t kc_rows, int rows) {
  if (kc_rows >= (int64_t(1) << 40) / (pl.d * 2)) return false;   // the strides a tensor map can have
  const uint64_t dims[3] = {static_cast<uint64_t>(pl.d), static_cast<uint64_t>(pl.H), static_cast<uint64_t>(pl.M)};
  const uint64_t strides[2] = {static_cast<uint64_t>(kc_rows) * pl.d * 2, static_cast<uint64_t>(pl.d) * 2};
  const uint32_t box[3] = {static_cast<uint32_t>(pl.d), static_cast<uint32_t>(pl.H), static_cast<uint32_t>(rows)};
  return make_tmap_bf16(tm, base, 3, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

cudaError_t launch_stream(const Plan& pl, int grid, const void* K, const void* V, void* Kc, void* Vc, int64_t kc_rows, int32_t* idx,
                          float* partials, const int32_t* slot_of_token, uint32_t* status, cudaStream_t st, bool* tmap_failed) {
  StreamArgs a;
  a.pl = pl;
  a.rule = make_window_rule(pl);
  a.K = static_cast<const uint8_t*>(K);
  a.V = static_cast<const uint8_t*>(V);
  a.Kc = static_cast<uint4*>(Kc);
  a.Vc = static_cast<uint4*>(Vc);
  a.kc_rows = kc_rows;
  a.rows = stream_rows(pl);
  a.idx = idx;
  a.slot_of_token = slot_of_token;
  a.partials = partials;
  a.status = status;
  CUtensorMap tm_kc = {}, tm_vc = {};
  if (pl.M > 0 && !(make_compact_tmap(&tm_kc, pl, Kc, kc_rows, 1) && make_compact_tmap(&tm_vc, pl, Vc, kc_rows, 1))) {
    *tmap_failed = true;
    return cudaSuccess;
  }
  const cudaError_t e = prepare_stream_kernels();
  if (e != cudaSuccess) return e;
  return launch_dependent(pl.H <= 16 ? build_kv_stream_kernel<1> : build_kv_stream_kernel<2>, grid, kStreamThreads, kStreamSmemBytes, st,
                          tm_kc, tm_vc, a);
}

cudaError_t launch_gather(const Plan& pl, int sm_count, const void* K, const void* V, void* Kc, void* Vc, int64_t kc_rows, int32_t* idx,
                          const int32_t* caller_idx, const int32_t* slot_of_token, uint32_t* status, float* zero_kmean, float* zero_vmean, cudaStream_t st,
                          bool* tmap_failed) {
  GatherArgs a;
  a.pl = pl;
  a.by_Lc = make_divisor(pl.Lc > 0 ? pl.Lc : 1);
  a.by_kept_w = make_divisor(pl.kept_w);
  a.K = static_cast<const uint8_t*>(K);
  a.V = static_cast<const uint8_t*>(V);
  a.Kc = static_cast<uint4*>(Kc);
  a.Vc = static_cast<uint4*>(Vc);
  a.kc_rows = kc_rows;
  a.stage_bytes = pl.H > 16 ? kGatherBytesManyHeads : kStreamBytes;
  a.rows = stream_rows(pl, a.stage_bytes);
  a.idx = idx;
  a.caller_idx = caller_idx;
  a.slot_of_token = slot_of_token;
  a.status = status;
  a.zero_kmean = zero_kmean;
  a.zero_vmean = zero_vmean;
  CUtensorMap tm_kc = {}, tm_vc = {};
  if (pl.M > 0 && !(make_compact_tmap(&tm_kc, pl, Kc, kc_rows, a.rows) && make_compact_tmap(&tm_vc, pl, Vc, kc_rows, a.rows))) {
    *tmap_failed = true;
    return cudaSuccess;
  }
  const cudaError_t e = prepare_stream_kernels();
  if (e != cudaSuccess) return e;
  const int64_t tiles = (pl.M + a.rows - 1) / a.rows, most = static_cast<int64_t>(sm_count) * (pl.H > 16 ? 1 : kStreamBlocks);
  const int grid = static_cast<int>(tiles < 1 ? 1 : tiles < most ? tiles : most);
  return launch_dependent(build_kv_gather_kernel, grid, 32, gather_smem_bytes(a.stage_bytes), st, tm_kc, tm_vc, a);
}

// Exchange buffer [n_ranks][2][H][slot_rows][d] (every rank's compact K then V, padded to slot_rows rows per
// head) -> Kc, Vc [H][M_total][d] with the ranks' rows one after the other.  One thread per 16-byte chunk.
struct ShardOffsets {
  int32_t n_ranks;
  int64_t first[kMaxShardRanks + 1];   // first compact row of rank r; first[n_ranks] = M_total
};
__global__ void __launch_bounds__(256)
assemble_shards_kernel(const uint4* __restrict__ gathered, const ShardOffsets off, const int H, const int64_t slot_rows,
                       uint4* __restrict__ Kc, uint4* __restrict__ Vc) {
  const int64_t m_total = off.first[off.n_ranks];
  const int64_t chunks = 2 * static_cast<int64_t>(H) * m_total * 8;   // 8 chunks of 16 bytes per row of 64 bf16
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < chunks;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t c = i & 7;
    int64_t row = i >> 3;                       // (which, head, m)
    const int64_t m = row % m_total;
    row /= m_total;
    const int64_t h = row % H;
    const int64_t which = row / H;
    int r = 0;
    while (r + 1 < off.n_ranks && m >= off.first[r + 1]) ++r;
    const int64_t src = ((((static_cast<int64_t>(r) * 2 + which) * H + h) * slot_rows) + (m - off.first[r])) * 8 + c;
    const uint4 v = gathered[src];
    (which == 0 ? Kc : Vc)[(h * m_total + m) * 8 + c] = v;
  }
}

}  // namespace

cudaError_t launch_assemble_shards(const void* gathered, int n_ranks, const int64_t* kept, int H, int d, int64_t slot_rows,
                                   void* Kc, void* Vc, const float* sums, int64_t n_dropped_total, float* kmean,
                                   float* vmean, cudaStream_t st) {
  ShardOffsets off;
  off.n_ranks = n_ranks;
  off.first[0] = 0;
  for (int r = 0; r < n_ranks; ++r) off.first[r + 1] = off.first[r] + kept[r];
  const int64_t chunks = 2 * static_cast<int64_t>(H) * off.first[n_ranks] * 8;
  if (chunks > 0) {
    int64_t blocks = (chunks + 255) / 256;
    if (blocks > 148 * 16) blocks = 148 * 16;
    assemble_shards_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(static_cast<const uint4*>(gathered), off, H, slot_rows,
                                                                         static_cast<uint4*>(Kc), static_cast<uint4*>(Vc));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (sums != nullptr && n_dropped_total > 0) {
    const int cols2 = 2 * H * d;
    mean_finalize_kernel<<<(cols2 + 31) / 32, 1024, 0, st>>>(sums, 1, cols2, 1.0f / static_cast<float>(n_dropped_total), kmean, vmean);
    return cudaGetLastError();
  }
  return cudaSuccess;
}

// Blocks per cluster of the few-token kernel: as many as leave one block per SM, up to 8; clusters of 8 find a place on at most
// three quarters of the SMs at once (8 heads, 16 clusters of 8: 7.6 us at 1,374 tokens, in two waves).
int small_ranks(const Plan& pl, int sm_count) {
  int ranks = 8;
  while (ranks > 1 && 2 * pl.H * ranks > (ranks == 8 ? sm_count * 3 / 4 : sm_count)) ranks /= 2;
  return ranks;
}

int build_kv_blocks_per_sm() { return kStreamBlocks; }

// Blocks of build_kv_stream_kernel.
int build_kv_grid(const Plan& pl, int sm_count) {
  const int rows = stream_rows(pl);
  const int64_t tiles = (pl.n_tok + rows - 1) / rows;
  const int64_t most = static_cast<int64_t>(sm_count) * build_kv_blocks_per_sm();
  return static_cast<int>(tiles < most ? tiles : most);
}

size_t build_kv_min_ws_bytes(const Plan& pl, int sm_count) {
  const int grid = build_kv_grid(pl, sm_count);
  const int64_t groups = (pl.n_tok + 7) / 8;
  const int64_t least = pl.H <= 16 ? grid : groups < sm_count ? groups : sm_count;
  return static_cast<size_t>(least < grid ? least : grid) * 2 * pl.H * pl.d * sizeof(float);
}

size_t build_kv_ws_bytes(const Plan& pl, int sm_count) {
  return static_cast<size_t>(build_kv_grid(pl, sm_count)) * 2 * pl.H * pl.d * sizeof(float);
}

cudaError_t launch_build_kv(const Plan& pl, int sm_count, const void* K, const void* V, void* Kc, void* Vc,
                            int32_t* idx, float* kmean, float* vmean, void* ws, size_t ws_bytes, cudaStream_t st,
                            bool* tmap_failed, const int32_t* caller_idx, int32_t* slot_of_token, int64_t kc_rows, bool sums_only,
                            void* clear_status) {
  *tmap_failed = false;
  if (kc_rows <= 0) kc_rows = pl.M;
  if (slot_of_token != nullptr) {
    // caller-chosen retained set: build the token -> compact position map first
    cudaError_t e0 = launch_dependent(fill_slots_kernel, static_cast<unsigned>((pl.n_tok + 255) / 256), 256, 0, st, slot_of_token, pl.n_tok);
    if (e0 == cudaSuccess && pl.M > 0 && caller_idx != nullptr)
      e0 = launch_dependent(scatter_slots_kernel, static_cast<unsigned>((pl.M + 255) / 256), 256, 0, st, caller_idx, pl.M, slot_of_token,
                            pl.n_tok);
    if (e0 != cudaSuccess) return e0;
    idx = nullptr;
  }
  const int ranks = small_ranks(pl, sm_count);
  if (pl.n_tok <= ranks * kSmallTokensPerBlock) {
    SmallArgs a;
    a.pl = pl;
    a.rule = make_window_rule(pl);
    a.K = static_cast<const uint4*>(K);
    a.V = static_cast<const uint4*>(V);
    a.Kc = static_cast<uint4*>(Kc);
    a.Vc = static_cast<uint4*>(Vc);
    a.kc_rows = kc_rows;
    a.idx = idx;
    a.slot_of_token = slot_of_token;
    a.kmean = pl.mean_fill != 0 ? kmean : nullptr;
    a.vmean = vmean;
    a.scale = pl.n_dropped <= 0 ? 0.f : sums_only ? 1.0f : 1.0f / static_cast<float>(pl.n_dropped);
    a.status = static_cast<uint32_t*>(clear_status);
    return launch_dependent_cluster(build_kv_small_kernel, 2 * pl.H * ranks, ranks, kSmallThreads, 0, st, a);
  }
  const int do_mean = (pl.mean_fill != 0 && pl.n_dropped > 0) ? 1 : 0;
  int grid = build_kv_grid(pl, sm_count);
  const size_t room = ws_bytes / (2 * static_cast<size_t>(pl.H) * pl.d * sizeof(float));   // partial rows
  if (do_mean && room < static_cast<size_t>(grid)) grid = static_cast<int>(room);
  float* partials = static_cast<float*>(ws);
  uint32_t* status = static_cast<uint32_t*>(clear_status);
  const bool zero_mean = pl.mean_fill != 0 && !do_mean;
  float* zk = zero_mean ? kmean : nullptr;
  float* zv = zero_mean ? vmean : nullptr;
  const cudaError_t e = do_mean ? launch_stream(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, slot_of_token, status, st, tmap_failed)
                                : launch_gather(pl, sm_count, K, V, Kc, Vc, kc_rows, idx, caller_idx, slot_of_token, status, zk, zv, st, tmap_failed);
  if (e != cudaSuccess || *tmap_failed || !do_mean) return e;
  const int cols2 = 2 * pl.H * pl.d;
  const float inv_count = sums_only ? 1.0f : 1.0f / static_cast<float>(pl.n_dropped);
  return launch_dependent(mean_finalize_kernel, (cols2 + 31) / 32, 1024, 0, st, partials, grid, cols2, inv_count, kmean, vmean);
}

}  // namespace avggt
