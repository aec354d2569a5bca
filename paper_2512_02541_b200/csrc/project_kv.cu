// K/V projection with the compaction of Sec. 4.3 fused into its epilogue:
//   K = X Wk^T + bk,  V = X Wv^T + bv        (bf16 operands, fp32 accumulation)
// and, while a tile of the result is still in tensor memory, the retained rows go to the
// head-major compact arrays, the dropped rows are added to the sums behind the mean pair, and
// (optionally) every row is written to the full K / V arrays.  The paper's remark that diagonal
// preservation and mean-fill cost "only O(N)" holds here without a second pass over K and V.
//
// A dense contraction, so it runs on the tensor cores: a persistent kernel of CTA pairs (clusters of two), one CTA per SM,
// a tile of 256 tokens x 256 output columns per pair.  A CTA holds its 128 tokens of X, half of the tile's rows of W and its
// 128 rows of the accumulator; the pair's products (cta_group::2) read W from both.  What bounds the single-CTA form of
// this kernel is shared memory: 48 KB written by TMA and read by the products per 64 channels, 768 clocks at 128 bytes per
// clock against 512 of the products.  The pair needs 32 KB, 512 clocks.  The epilogue then had to become lighter as well (10,700 clocks a tile against 7,800 of the
// products): column sums kept per lane instead of 124 shuffles a tile, biases from shared memory, window rule without
// divisions, the accumulator released after its last read.  137,400 tokens x 1024 -> 2 x 1024, full K and V written:
// 571 -> 502 us (1010 -> 1147 TFLOP/s).
//   warp 0      TMA producer: X tiles (128 tokens x 64 channels) and half W tiles (128 output columns x
//               64 channels) through a six-stage shared-memory ring (128-byte swizzle); the copies of both CTAs
//               signal the even CTA's barrier
//   warp 1      MMA issuer (even CTA): tcgen05.mma, M 256 x N 256 x K 16, fp32 accumulators in tensor memory;
//               two accumulators of 256 columns, so the next tile's products run under this
//               tile's epilogue
//   warp 2      hands a read accumulator back to the even CTA
//   warps 4-11  epilogue, one token row and half of the tile's columns per thread: accumulator -> registers, bias, bf16; a head's
//               64 values of the warp's 32 rows are staged in shared memory (128-byte swizzle),
//               from where one TMA store writes them to the full K / V array and the retained
//               rows are copied, 128 contiguous bytes at a time, to the compact arrays (a thread
//               storing its own row 16 bytes at a time kept the store path busy for longer than
//               the products of the tile take);
//               each lane adds up its own dropped rows, column by column, in registers for all the tiles of the CTA,
//               and the 32 lanes come together once at the end (a transposing shuffle reduction: lane c ends up with
//               column c)
// A pair keeps one block of 256 output columns (four heads of K or of V) for its whole life and
// walks over token tiles; pairs with the same token tile run side by side, so an X tile is
// fetched from HBM once and from L2 by the others.  Per-CTA partial sums go to the workspace and
// a small second kernel adds them in a fixed order: no floating-point atomics, results identical
// from run to run.
#include <cstddef>
#include <mutex>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"
#include "tmap.h"

namespace avggt {

namespace {

constexpr int kTileTok = 128;     // token rows per CTA
constexpr int kPairTok = 2 * kTileTok;   // per tile (M of the MMA)
constexpr int kTileCol = 256;     // output columns per tile (N of the MMA): four heads of 64
constexpr int kBlockK = 64;       // channels per ring stage: one 128-byte swizzle row
constexpr int kProjStages = 6;
constexpr uint32_t kBytesA = kTileTok * kBlockK * 2;   // 16 KiB
constexpr uint32_t kBytesB = kTileCol / 2 * kBlockK * 2;   // 16 KiB: a CTA's half
constexpr uint32_t kStageBytes = 32 * 128;   // epilogue staging: 32 rows x one head (64 bf16), one per epilogue warp
constexpr int kEpiWarps = 8;        // warps 4..11: warp % 4 is the lane quarter of tensor memory, (warp - 4) / 4 the half of
                                    // the tile's 256 columns (two heads each)
constexpr int kFirstEpiWarp = 4;    // warp 3 is idle: it completes the first warpgroup, so that registers can be moved
constexpr int kProjThreads = 32 * (kFirstEpiWarp + kEpiWarps);
// Registers per thread after the roles have split (an epilogue thread keeps 128 column sums).  The sum over all warps must not
// exceed what the launch allocated, or setmaxnreg.inc waits for ever: prepare_kernel refuses a build that allocates less.
constexpr int kRegsEpi = 216, kRegsIssue = 40;
constexpr int kRegsTotal = kRegsEpi * kEpiWarps + kRegsIssue * kFirstEpiWarp;
constexpr uint32_t kProjTmemCols = 512;

struct ProjArgs {
  Plan pl;
  WindowRule rule;
  int32_t C;              // model dimension (channels of X)
  int32_t n_col_tiles;    // column tiles of one projection: ceil(H * d / 256)
  int32_t n_tok_tiles;    // ceil(n_tok / 256)
  int32_t tok_stride;     // token tiles a pair advances by: pairs / (2 * n_col_tiles)
  const float* bias_k;    // [H * d] or null
  const float* bias_v;
  uint4* K_full;          // [n_tok, H, d] or null
  uint4* V_full;
  uint4* Kc;              // [H, M, d]
  uint4* Vc;
  int32_t* idx;           // [M] or null
  float* partials;        // [gridDim.x][4 warps][256]: sums over the dropped rows this warp has seen
  uint32_t* status;       // 4 words, as in the attention kernel
  int32_t do_mean;
  int32_t zero_means;     // zero-fill kmean and vmean
  float* kmean;
  float* vmean;
};

struct __align__(8) ProjBarriers {
  uint64_t full[kProjStages];    // even CTA's: both CTAs' copies of the stage have landed
  uint64_t empty[kProjStages];   // either CTA's own: the products have read the stage
  uint64_t acc_full[2];          // either CTA's own: the tile's products have completed
  uint64_t acc_read[2];          // either CTA's own: its epilogue warps have read the accumulator
  uint64_t acc_empty[2];         // even CTA's: those of both CTAs have (one arrival from each, see warp 2)
  uint64_t mma_idle;             // MMA issuer -> itself: every product it issued has completed
  uint32_t tmem_base;
  uint32_t abort_flag;
};

__device__ __forceinline__ void proj_report(const ProjArgs& a, ProjBarriers* bars, uint32_t where, uint32_t iter) {
  if (atomicCAS(a.status, 0u, 1u) == 0u) {
    a.status[1] = blockIdx.x;
    a.status[2] = where;
    a.status[3] = iter;
  }
  *reinterpret_cast<volatile uint32_t*>(&bars->abort_flag) = 1u;
}

// Bounded wait; false when the limit ran out or another role of the CTA gave up.
__device__ __forceinline__ bool proj_wait(uint64_t* bar, uint32_t parity, ProjBarriers* bars, const ProjArgs& a,
                                          uint32_t where, uint32_t iter, bool check_abort = true) {
  const uint32_t b = smem_u32(bar);
  if (mbar_try_wait_cluster(b, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  uint32_t spins = 0;
  while (true) {
    if (mbar_try_wait_cluster(b, parity)) return true;
    if ((++spins & 0xffu) == 0) {
      if (check_abort && *reinterpret_cast<volatile uint32_t*>(&bars->abort_flag)) return false;
      if (globaltimer_ns() - t0 > AVGGT_WAIT_LIMIT_NS) {
        proj_report(a, bars, where, iter);
        return false;
      }
    }
  }
}
__device__ __forceinline__ bool proj_wait_warp(uint64_t* bar, uint32_t parity, ProjBarriers* bars, const ProjArgs& a,
                                               uint32_t where, uint32_t iter, bool check_abort = true) {
  return __all_sync(0xffffffffu, proj_wait(bar, parity, bars, a, where, iter, check_abort));
}

// v[i] of lane l  ->  lane c returns sum over l of v[c] (of lane l): 31 shuffles for 32 columns.
__device__ __forceinline__ float warp_column_sums(float (&v)[32], int lane) {
#pragma unroll
  for (int half = 16; half >= 1; half >>= 1) {
    // lanes with the bit set keep the upper `half` entries, the others the lower ones
    const bool upper = (lane & half) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const float mine = upper ? v[i + half] : v[i];
      const float theirs = upper ? v[i] : v[i + half];
      v[i] = mine + __shfl_xor_sync(0xffffffffu, theirs, half);
    }
  }
  return v[0];
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kProjThreads, 1)
project_kv_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_wk,
                  const __grid_constant__ CUtensorMap tm_wv, const __grid_constant__ CUtensorMap tm_kfull,
                  const __grid_constant__ CUtensorMap tm_vfull, const ProjArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;                               // kProjStages tiles of X
  uint8_t* sB = smem + kProjStages * kBytesA;       // kProjStages tiles of W
  uint8_t* sStage = sB + kProjStages * kBytesB;     // one staging tile per epilogue warp
  __shared__ ProjBarriers bars;
  __shared__ uint8_t kept_rows[kEpiWarps][32];   // an epilogue warp's retained rows, in order
  __shared__ __align__(16) float bias_cols[kTileCol];   // of this CTA's block of output columns

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_cta_rank();     // 0: the even CTA, which issues the products
  const int pair = blockIdx.x >> 1;
  // this pair's block of output columns, for its whole life
  const int col_tile_all = pair % (2 * a.n_col_tiles);
  const int which = col_tile_all / a.n_col_tiles;                 // 0: K, 1: V
  const int col_tile = col_tile_all - which * a.n_col_tiles;
  const int tok0 = pair / (2 * a.n_col_tiles);                    // first token tile
  const int n_kb = a.C / kBlockK;

  // a thread for each barrier (one alone takes hundreds of clocks for them)
  constexpr int kBarriers = static_cast<int>(offsetof(ProjBarriers, tmem_base) / sizeof(uint64_t));
  constexpr int kAccRead = static_cast<int>(offsetof(ProjBarriers, acc_read) / sizeof(uint64_t));
  if (threadIdx.x < kBarriers) {
    const int which_bar = static_cast<int>(threadIdx.x) - kAccRead;
    mbar_init(smem_u32(&bars) + threadIdx.x * sizeof(uint64_t), which_bar == 0 || which_bar == 1 ? kEpiWarps : which_bar == 2 || which_bar == 3 ? 2 : 1);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) bars.abort_flag = 0;
  if (warp == 0) {
    tmem_alloc_pair(smem_u32(&bars.tmem_base), kProjTmemCols);
    tmem_relinquish_pair();
  }
  // everything above may run while the kernel before this one ends
  grid_dependency_wait();
  for (int c = threadIdx.x; c < kTileCol; c += kProjThreads) {
    const float* b = which == 0 ? a.bias_k : a.bias_v;
    const int col = col_tile * kTileCol + c;
    bias_cols[c] = b != nullptr && col < a.pl.H * a.pl.d ? b[col] : 0.f;
  }
  if (blockIdx.x == 0 && a.zero_means && threadIdx.x < 256) {   // a problem that drops nothing
    for (int i = threadIdx.x; i < a.pl.H * a.pl.d; i += 256) { a.kmean[i] = 0.f; a.vmean[i] = 0.f; }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // the other CTA's barriers are initialised
  tc_fence_after();
  const uint32_t tmem = bars.tmem_base;

  if (warp < kFirstEpiWarp) {
    reg_dec<kRegsIssue>();
    if (warp == 0) {
      // ------------------------------------------------------------ TMA producer
      const CUtensorMap* tm_w = which == 0 ? &tm_wk : &tm_wv;
      if (elect_one()) {
        prefetch_tensormap(&tm_x);
        prefetch_tensormap(tm_w);
      }
      int stage = 0, issued = 0;
      uint32_t parity = 1;   // a fresh barrier passes the wait on the "previous" phase at once
      bool ok = true;
      for (int tt = tok0; tt < a.n_tok_tiles && ok; tt += a.tok_stride) {
        for (int kb = 0; kb < n_kb; ++kb) {
          ok = proj_wait_warp(&bars.empty[stage], parity, &bars, a, 10, issued);
          if (!ok) break;
          if (elect_one()) {
            const uint32_t fb = smem_u32(&bars.full[stage]);
            if (rank == 0) mbar_arrive_expect_tx(fb, 2 * (kBytesA + kBytesB));
            const uint32_t even = cluster_addr(fb, 0);
            tma_load_2d_pair(smem_u32(sA + stage * kBytesA), &tm_x, kb * kBlockK, tt * kPairTok + static_cast<int>(rank) * kTileTok, even);
            tma_load_2d_pair(smem_u32(sB + stage * kBytesB), tm_w, kb * kBlockK,
                             col_tile * kTileCol + static_cast<int>(rank) * (kTileCol / 2), even);
          }
          __syncwarp();
          ++issued;
          if (++stage == kProjStages) { stage = 0; parity ^= 1; }
        }
      }
      // let the copies in flight land before the pair gives up its shared memory (the even CTA waits for both)
      if (!ok && rank == 0) {
        for (int back = 1; back <= kProjStages; ++back) {
          const int jt = issued - back;
          if (jt >= 0) (void)proj_wait_warp(&bars.full[jt % kProjStages], (jt / kProjStages) & 1, &bars, a, 12, jt, false);
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------ MMA issuer (even CTA)
      constexpr uint32_t idesc = umma_idesc_bf16(kPairTok, kTileCol, false);
      constexpr uint16_t both = 3;
      int stage = 0, it = 0;
      uint32_t parity = 0;
      bool ok = true;
      for (int tt = tok0; rank == 0 && tt < a.n_tok_tiles && ok; tt += a.tok_stride, ++it) {
        const int buf = it & 1;
        // the epilogue has emptied this accumulator (first use of either buffer: passes at once)
        ok = proj_wait_warp(&bars.acc_empty[buf], ((it >> 1) & 1) ^ 1, &bars, a, 20, it);
        if (!ok) break;
        tc_fence_after();
        for (int kb = 0; kb < n_kb; ++kb) {
          ok = proj_wait_warp(&bars.full[stage], parity, &bars, a, 21, kb);
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t da = umma_desc_lo(smem_u32(sA + stage * kBytesA), 16);
            const uint32_t db = umma_desc_lo(smem_u32(sB + stage * kBytesB), 16);
  #pragma unroll
            for (int k = 0; k < kBlockK / 16; ++k)
              umma_ss_pair(tmem + buf * kTileCol, da + (k * 32 >> 4), db + (k * 32 >> 4), idesc, kb > 0 || k > 0);
            umma_commit_pair(smem_u32(&bars.empty[stage]), both);
            if (kb == n_kb - 1) umma_commit_pair(smem_u32(&bars.acc_full[buf]), both);
          }
          __syncwarp();
          if (++stage == kProjStages) { stage = 0; parity ^= 1; }
        }
      }
      // every product this warp issued has completed before tensor memory is freed (also on a wait that ran out)
      __syncwarp();
      if (rank == 0) {
        if (elect_one()) umma_commit_pair(smem_u32(&bars.mma_idle), 1);
        __syncwarp();
        (void)proj_wait_warp(&bars.mma_idle, 0, &bars, a, 22, it, false);
      }
    } else if (warp == 2) {
      // ------------------------------------------------------------ hands the accumulators back to the even CTA
      // An arrival on the other CTA's barrier that releases what came before it waits until the thread's stores to global memory have
      // completed (some 2,000 clocks in the epilogue).  So the epilogue warps arrive on their own CTA's barrier, and this warp, which
      // stores nothing, passes the arrival on.
      int it = 0;
      for (int tt = tok0; tt < a.n_tok_tiles; tt += a.tok_stride, ++it) {
        const int buf = it & 1;
        if (!proj_wait_warp(&bars.acc_read[buf], (it >> 1) & 1, &bars, a, 31, it)) break;
        tc_fence_after();
        tc_fence_before();
        if (elect_one()) mbar_arrive_cluster(cluster_addr(smem_u32(&bars.acc_empty[buf]), 0));
        __syncwarp();
      }
    }
  } else {
    reg_inc<kRegsEpi>();
    // ------------------------------------------------------------ epilogue: one token row per thread
    const Plan& pl = a.pl;
    const int quarter = warp & 3;                       // tensor-memory lanes [32 quarter, 32 quarter + 32)
    const int col_half = (warp - kFirstEpiWarp) >> 2;               // columns [128 col_half, 128 col_half + 128) of the tile
    uint8_t* sbuf = sStage + (warp - kFirstEpiWarp) * kStageBytes;
    const bool write_full = (which == 0 ? a.K_full : a.V_full) != nullptr;
    const CUtensorMap* tm_full = which == 0 ? &tm_kfull : &tm_vfull;
    uint4* compact = which == 0 ? a.Kc : a.Vc;
    const int cols_total = pl.H * pl.d;
    // This lane's part of the sums of columns 128 col_half .. + 127 over dropped rows (pairs of columns).  Each lane adds up its
    // own rows for all the tiles of the CTA; the lanes come together once, at the end.
    uint64_t colsum[64];
#pragma unroll
    for (int i = 0; i < 64; ++i) colsum[i] = pack_f32x2(0.f, 0.f);
    // this warp's 128 biases, read back 16 bytes at a time
    float* sbias = bias_cols + 128 * col_half;
    int it = 0;
    bool ok = true;
    for (int tt = tok0; tt < a.n_tok_tiles; tt += a.tok_stride, ++it) {
      const int buf = it & 1;
      ok = proj_wait_warp(&bars.acc_full[buf], (it >> 1) & 1, &bars, a, 30, it);
      if (!ok) break;
      tc_fence_after();
      const int64_t row0 = static_cast<int64_t>(tt) * kPairTok + rank * kTileTok + quarter * 32;   // first row of this warp
      const int64_t row = row0 + lane;
      const bool row_valid = row < pl.n_tok;
      const int32_t m = row_valid ? compact_position(a.rule, pl, static_cast<uint32_t>(row)) : -1;
      const bool kept = m >= 0;
      const bool dropped = row_valid && m < 0;
      if (kept && which == 0 && col_tile == 0 && col_half == 0 && a.idx != nullptr) a.idx[m] = static_cast<int32_t>(row);
      const uint32_t kept_mask = __ballot_sync(0xffffffffu, kept);
      const int n_kept = __popc(kept_mask);
      __syncwarp();   // the previous tile's list has been read
      if (kept) kept_rows[warp - kFirstEpiWarp][__popc(kept_mask & ((1u << lane) - 1))] = static_cast<uint8_t>(lane);
      __syncwarp();
      const uint32_t t_acc = tmem + buf * kTileCol + (static_cast<uint32_t>(32 * quarter) << 16);
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {                              // one head (64 columns) at a time
        const int hg = 2 * col_half + hh;                           // head within the tile
        const int col0 = col_tile * kTileCol + hg * 64;             // first column within K (or V)
        if (col0 >= cols_total) break;                              // warp-uniform: H * d is a multiple of 64
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          uint32_t raw[32];
          tmem_ld32(t_acc + hg * 64 + half * 32, raw);
          tmem_wait_ld();
          if (hh == 1 && half == 1) {   // this warp is done with the accumulator
            tc_fence_before();
            if (elect_one()) mbar_arrive(smem_u32(&bars.acc_read[buf]));
          }
          uint64_t v[16];
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 b = *reinterpret_cast<const float4*>(sbias + hh * 64 + half * 32 + 4 * i);
            v[2 * i] = add_f32x2(pack_f32x2(__uint_as_float(raw[4 * i]), __uint_as_float(raw[4 * i + 1])), pack_f32x2(b.x, b.y));
            v[2 * i + 1] = add_f32x2(pack_f32x2(__uint_as_float(raw[4 * i + 2]), __uint_as_float(raw[4 * i + 3])), pack_f32x2(b.z, b.w));
          }
          if (half == 0) {
            // the store of the previous head has finished reading the staging tile
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
          }
          // row `lane` of the staging tile, 16-byte chunks 4 half .. 4 half + 3, swizzled as TMA expects them
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint4 o;
            o.x = pack_bf16x2(v[4 * i]);
            o.y = pack_bf16x2(v[4 * i + 1]);
            o.z = pack_bf16x2(v[4 * i + 2]);
            o.w = pack_bf16x2(v[4 * i + 3]);
            *reinterpret_cast<uint4*>(sbuf + lane * 128 + (((4 * half + i) ^ (lane & 7)) << 4)) = o;
          }
          if (a.do_mean && dropped) {
#pragma unroll
            for (int i = 0; i < 16; ++i) colsum[(2 * hh + half) * 16 + i] = add_f32x2(colsum[(2 * hh + half) * 16 + i], v[i]);
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        // every row of the tile to the full array (rows beyond the last token are clipped by the tensor map)
        if (write_full && lane == 0) {
          tma_store_2d(tm_full, smem_u32(sbuf), col0, static_cast<int>(row0));
          bulk_commit();
        }
        // retained rows to the compact array: four rows per pass, eight lanes x 16 bytes per row
        const int head = col0 >> 6;
        for (int k0 = 0; k0 < n_kept; k0 += 4) {
          const int k = k0 + (lane >> 3);
          const bool have = k < n_kept;
          const int r = have ? kept_rows[warp - kFirstEpiWarp][k] : 0;
          const int32_t m_r = __shfl_sync(0xffffffffu, m, r);
          if (have) {
            const uint4 val = *reinterpret_cast<const uint4*>(sbuf + r * 128 + (((lane & 7) ^ (r & 7)) << 4));
            compact[(static_cast<size_t>(head) * static_cast<size_t>(pl.M) + static_cast<size_t>(m_r)) * 8 + (lane & 7)] = val;
          }
        }
      }
      if (2 * col_half * 64 + 64 + col_tile * kTileCol >= cols_total) {   // a second head (or both) beyond the last: not reached above
        tc_fence_before();
        if (elect_one()) mbar_arrive(smem_u32(&bars.acc_read[buf]));
      }
    }
    if (lane == 0) bulk_wait_read<0>();   // the staging tiles stay put until the last store has read them
    __syncwarp();
    if (ok && a.do_mean) {
      float* dst = a.partials + (static_cast<size_t>(blockIdx.x) * 4 + quarter) * kTileCol + 128 * col_half;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float v[32];
#pragma unroll
        for (int c = 0; c < 16; ++c) unpack_f32x2(colsum[16 * i + c], v[2 * c], v[2 * c + 1]);
        dst[32 * i + lane] = warp_column_sums(v, lane);
      }
    }
  }

  grid_launch_dependents();
  tmem_wait_ld();
  tc_fence_before();
  __syncthreads();
  cluster_sync();   // neither CTA leaves, or gives up tensor memory, while the other may still signal it or compute in it
  tc_fence_after();
  if (warp == 0) tmem_dealloc_pair(tmem, kProjTmemCols);
}

// kmean[col] = (sum over the CTAs that own col's block, and their four epilogue warps, in a fixed order) / n_dropped
__global__ void __launch_bounds__(256)
project_mean_kernel(const float* partials, int grid, int n_col_tiles, int cols_total, float inv_count,
                    float* __restrict__ kmean, float* __restrict__ vmean) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int g = blockIdx.x * blockDim.x + threadIdx.x;     // column of [K | V]
  if (g >= 2 * cols_total) return;
  const int which = g / cols_total, col = g - which * cols_total;
  const int col_tile_all = which * n_col_tiles + col / kTileCol, in_tile = col % kTileCol;
  float s = 0.f;
  for (int pair = col_tile_all; pair < grid / 2; pair += 2 * n_col_tiles)
    for (int w = 0; w < 8; ++w) s += __ldcg(partials + (static_cast<size_t>(pair) * 8 + w) * kTileCol + in_tile);   // both CTAs' four
  (which == 0 ? kmean : vmean)[col] = s * inv_count;
}

constexpr size_t kProjSmemBytes = static_cast<size_t>(kProjStages) * (kBytesA + kBytesB) + 8 * kStageBytes + 1024;

// Once per device: the register check (see kRegsTotal) and the dynamic shared-memory limit of the kernel.
cudaError_t prepare_kernel() {
  static std::mutex mu;
  static bool ready[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!ready[dev]) {
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, project_kv_kernel);
    if (e != cudaSuccess) return e;
    if (fa.numRegs * (kProjThreads / 32) < kRegsTotal) return cudaErrorLaunchOutOfResources;
    e = cudaFuncSetAttribute(project_kv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kProjSmemBytes));
    if (e != cudaSuccess) return e;
    ready[dev] = true;
  }
  return cudaSuccess;
}

int project_grid(const Plan& pl, int sm_count) {
  const int per_tok = 2 * ((pl.H * pl.d + kTileCol - 1) / kTileCol);
  int pairs = (sm_count / 2 / per_tok) * per_tok;
  if (pairs < per_tok) pairs = per_tok;
  const int64_t tok_tiles = (pl.n_tok + kPairTok - 1) / kPairTok;
  if (pairs / per_tok > tok_tiles) pairs = static_cast<int>(tok_tiles) * per_tok;
  const int g = 2 * pairs;
  return g;
}

}  // namespace

size_t project_kv_ws_bytes(const Plan& pl, int sm_count) {
  return kAttnStatusBytes + static_cast<size_t>(project_grid(pl, sm_count)) * 4 * kTileCol * sizeof(float);
}

cudaError_t launch_project_kv(const Plan& pl, int sm_count, int model_dim, const void* X, const void* Wk, const void* Wv,
                              const float* bias_k, const float* bias_v, void* K, void* V, void* Kc, void* Vc, int32_t* idx,
                              float* kmean, float* vmean, void* ws, cudaStream_t st, bool* tmap_failed) {
  *tmap_failed = false;
  const int cols_total = pl.H * pl.d;
  ProjArgs a;
  a.pl = pl;
  a.rule = make_window_rule(pl);
  a.C = model_dim;
  a.n_col_tiles = (cols_total + kTileCol - 1) / kTileCol;
  a.n_tok_tiles = static_cast<int32_t>((pl.n_tok + kPairTok - 1) / kPairTok);
  const int grid = project_grid(pl, sm_count);
  a.tok_stride = grid / 2 / (2 * a.n_col_tiles);
  a.bias_k = bias_k;
  a.bias_v = bias_v;
  a.K_full = static_cast<uint4*>(K);
  a.V_full = static_cast<uint4*>(V);
  a.Kc = static_cast<uint4*>(Kc);
  a.Vc = static_cast<uint4*>(Vc);
  a.idx = idx;
  a.status = static_cast<uint32_t*>(ws);
  a.partials = reinterpret_cast<float*>(static_cast<char*>(ws) + kAttnStatusBytes);
  a.do_mean = (pl.mean_fill != 0 && pl.n_dropped > 0) ? 1 : 0;
  a.zero_means = pl.mean_fill != 0 && !a.do_mean;
  a.kmean = kmean;
  a.vmean = vmean;

  CUtensorMap tm_x, tm_wk, tm_wv, tm_kfull, tm_vfull;
  const uint64_t x_dims[2] = {static_cast<uint64_t>(model_dim), static_cast<uint64_t>(pl.n_tok)};
  const uint64_t w_dims[2] = {static_cast<uint64_t>(model_dim), static_cast<uint64_t>(cols_total)};
  const uint64_t row_bytes[1] = {static_cast<uint64_t>(model_dim) * 2};
  const uint32_t x_box[2] = {kBlockK, kTileTok};
  const uint32_t w_box[2] = {kBlockK, kTileCol / 2};
  bool good = make_tmap_bf16(&tm_x, X, 2, x_dims, row_bytes, x_box);
  good = good && make_tmap_bf16(&tm_wk, Wk, 2, w_dims, row_bytes, w_box);
  good = good && make_tmap_bf16(&tm_wv, Wv, 2, w_dims, row_bytes, w_box);
  // the full K / V arrays as [n_tok, H * d], written 32 rows x one head at a time (any valid map stands in for an
  // array that is not wanted; the kernel does not use it then)
  const uint64_t f_dims[2] = {static_cast<uint64_t>(cols_total), static_cast<uint64_t>(pl.n_tok)};
  const uint64_t f_row_bytes[1] = {static_cast<uint64_t>(cols_total) * 2};
  const uint32_t f_box[2] = {64, 32};
  if (K != nullptr) good = good && make_tmap_bf16(&tm_kfull, K, 2, f_dims, f_row_bytes, f_box);
  else tm_kfull = tm_x;
  if (V != nullptr) good = good && make_tmap_bf16(&tm_vfull, V, 2, f_dims, f_row_bytes, f_box);
  else tm_vfull = tm_x;
  if (!good) { *tmap_failed = true; return cudaSuccess; }

  cudaError_t e = prepare_kernel();
  if (e == cudaSuccess) e = launch_clear_status(ws, st);
  if (e == cudaSuccess)
    e = launch_dependent(project_kv_kernel, grid, kProjThreads, kProjSmemBytes, st, tm_x, tm_wk, tm_wv, tm_kfull, tm_vfull, a);
  if (e == cudaSuccess && a.do_mean)
    e = launch_dependent(project_mean_kernel, (2 * cols_total + 255) / 256, 256, 0, st, a.partials, grid, a.n_col_tiles, cols_total,
                         1.0f / static_cast<float>(pl.n_dropped), kmean, vmean);
  return e;
}

}  // namespace avggt
