// K/V compaction and mean-fill reduction (Sec. 4.3 of the AVGGT paper):
// one pass over K and V that copies the retained rows into the head-major
// compact arrays and sums the dropped patch rows for the mean Key/Value pair.
//
// Memory-bound: every row of K and V is read once with 16-byte loads (a warp
// covers 512 contiguous bytes per load instruction), retained rows are written
// once as full 128-byte lines.  Sums are kept in registers per lane (a lane owns
// fixed columns), reduced across the warps of a block in shared memory in a
// fixed order, written as one partial row per block, and reduced across blocks
// by a second small kernel with a fixed shuffle tree: no floating-point
// atomics, so the result does not change from run to run.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "internal.h"
#include "ptx.cuh"

namespace avggt {

namespace {

constexpr int kBuildThreads = 256;
constexpr int kBuildWarps = kBuildThreads / 32;
// Blocks of build_kv_kernel<PASSES> that an SM holds (by its registers; the launch bounds see to it that they fit), and as many as
// the grid has per SM: a second wave of blocks would only double the partial sums (592 blocks instead of 296 on 148 SMs: 16.2 instead of 13.5 us at 8 frames,
// 30.8 instead of 27.7 at 24; no difference at 333).
constexpr int kBuildBlocks[9] = {0, 5, 3, 2, 2, 1, 1, 1, 1};

// The kernels here begin while the kernel before them in the stream, and one before that which has already let it begin, may still
// be writing what they read after their wait: K and V (the projection), the map from tokens to compact positions, a caller's
// list of retained tokens.  They therefore read none of it by the read-only path, which is for data that does not change in a
// kernel's lifetime, or through a pointer the compiler may take for one to such data: K and V by this load, the rest by __ldcg.
// (The compaction of 333 frames takes the same time with either load, 396 us.)
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

// PASSES = ceil(H * 8 / 32): 16-byte chunks of one row handled per lane.
// kc_rows: rows per head of the compact arrays (M, or more when the caller's arrays are a slot of a
// larger exchange buffer).
template <int PASSES>
__global__ void __launch_bounds__(kBuildThreads, kBuildBlocks[PASSES])
build_kv_kernel(const Plan pl, const uint4* K, const uint4* V, uint4* __restrict__ Kc,
                uint4* __restrict__ Vc, const int64_t kc_rows, int32_t* __restrict__ idx, float* __restrict__ partials,
                const int do_mean, const int32_t* slot_of_token, uint32_t* __restrict__ status,
                float* __restrict__ zero_kmean, float* __restrict__ zero_vmean) {
  extern __shared__ float red[];   // [kBuildWarps][PASSES * 256]
  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const uint32_t chunks_per_row = static_cast<uint32_t>(pl.H) * 8u;   // 16-byte chunks (d = 64 bf16 = 8 chunks per head)
  const uint32_t n_tok = static_cast<uint32_t>(pl.n_tok);
  const uint32_t warps_total = gridDim.x * kBuildWarps;

  grid_dependency_wait();
  if (blockIdx.x == 0) {
    // what would otherwise be launches of their own: the status block of the attention that follows, and the mean pair of
    // a problem that drops nothing
    if (status != nullptr && threadIdx.x < kAttnStatusBytes / 4) status[threadIdx.x] = 0u;
    if (zero_kmean != nullptr)
      for (int i = threadIdx.x; i < pl.H * pl.d; i += kBuildThreads) { zero_kmean[i] = 0.f; zero_vmean[i] = 0.f; }
  }

  float acc_k[PASSES][8], acc_v[PASSES][8];
#pragma unroll
  for (int p = 0; p < PASSES; ++p)
#pragma unroll
    for (int e = 0; e < 8; ++e) { acc_k[p][e] = 0.f; acc_v[p][e] = 0.f; }

  for (uint32_t row = blockIdx.x * kBuildWarps + warp; row < n_tok; row += warps_total) {
    const int32_t f = static_cast<int32_t>(row / static_cast<uint32_t>(pl.L));
    const int32_t u = static_cast<int32_t>(row - static_cast<uint32_t>(f) * static_cast<uint32_t>(pl.L));
    // compact position within the frame's block by the window rule, or, for a caller-chosen retained set,
    // the global compact position from the caller's map
    const int32_t cs = slot_of_token != nullptr ? __ldcg(slot_of_token + row) : compact_slot(pl, f, u);
    if (cs < 0 && !do_mean) continue;
    const uint4* krow = K + static_cast<size_t>(row) * chunks_per_row;
    const uint4* vrow = V + static_cast<size_t>(row) * chunks_per_row;
    uint4 kv[PASSES], vv[PASSES];
#pragma unroll
    for (int p = 0; p < PASSES; ++p) {
      const uint32_t c = p * 32 + lane;
      if (c < chunks_per_row) { kv[p] = ld_stream(krow + c); vv[p] = ld_stream(vrow + c); }
      else { kv[p] = make_uint4(0, 0, 0, 0); vv[p] = make_uint4(0, 0, 0, 0); }
    }
    if (cs >= 0) {
      const int64_t m = slot_of_token != nullptr ? cs : compact_frame_base(pl, f) + cs;
      if (lane == 0 && idx != nullptr) idx[m] = static_cast<int32_t>(row);
#pragma unroll
      for (int p = 0; p < PASSES; ++p) {
        const uint32_t c = p * 32 + lane;
        if (c < chunks_per_row) {
          const size_t dst = (static_cast<size_t>(c >> 3) * static_cast<size_t>(kc_rows) + static_cast<size_t>(m)) * 8u + (c & 7u);
          Kc[dst] = kv[p];
          Vc[dst] = vv[p];
        }
      }
    } else {
#pragma unroll
      for (int p = 0; p < PASSES; ++p) { add_bf16x8(acc_k[p], kv[p]); add_bf16x8(acc_v[p], vv[p]); }
    }
  }

  // the next kernel may take its place on the chip while the blocks reduce and end (earlier it would only be in the way)
  grid_launch_dependents();
  if (!do_mean) return;
  // block reduction, K then V, fixed order over warps
  const int cols = pl.H * pl.d;   // = chunks_per_row * 8
#pragma unroll
  for (int which = 0; which < 2; ++which) {
    float* mine = red + warp * (PASSES * 256);
#pragma unroll
    for (int p = 0; p < PASSES; ++p)
#pragma unroll
      for (int e = 0; e < 8; ++e) mine[(p * 32 + lane) * 8 + e] = which == 0 ? acc_k[p][e] : acc_v[p][e];
    __syncthreads();
    for (int col = threadIdx.x; col < cols; col += kBuildThreads) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < kBuildWarps; ++w) s += red[w * (PASSES * 256) + col];
      partials[static_cast<size_t>(blockIdx.x) * (2 * cols) + which * cols + col] = s;
    }
    __syncthreads();
  }
}

// The same for few tokens, in one launch: a cluster of thread blocks takes one head of K or of V, each block every
// cluster-size-th group of 128 rows, and adds the blocks' sums up through distributed shared memory.  No partial sums in
// global memory (for a few frames as many bytes as K and V themselves) and no second kernel.  A row's 128 bytes of the
// head are read by 8 threads, 16 bytes each, four rows in flight per thread.
constexpr int kSmallThreads = 1024;
constexpr int kSmallRows = kSmallThreads / 8;   // rows a block reads at once

// Up to so many tokens per block of a cluster.  Above, the bytes are the bound, which more blocks per SM and warps that read
// whole rows serve better.  The two kernels' times in us, this one first (148 SMs): 16 heads, clusters of 4, limit 5,760:
// 4.5 and 6.2 at 1,374 tokens, 7.9 and 10.4 at 4,122, 10.3 and 12.0 at 5,496, 16.2 and 14.1 at 8,244.  6 heads, clusters of 8,
// limit 11,520: 4.2 and 4.9 at 1,374, 6.0 and 8.8 at 5,496, 9.1 and 11.3 at 10,992, 19.8 and 17.9 at 21,984.  24 heads, clusters
// of 2, limit 2,880: 5.9 and 8.6 at 1,374.  Of 261 tokens and up to 8 heads it is 0.4 us slower (3.7 and 3.3) and saves
// the host a launch.
constexpr int64_t kSmallTokensPerBlock = 1440;

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
  __shared__ float part[64];   // this block's sums, read by the cluster's first block
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
  if (threadIdx.x < 64) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kSmallThreads / 32; ++w) s += red[w][threadIdx.x];
    part[threadIdx.x] = s;
  }
  cluster_sync();
  if (rank == 0 && threadIdx.x < 64) {
    float s = 0.f;
    for (uint32_t r = 0; r < n_ranks; ++r) s += ld_cluster_f32(cluster_addr(smem_u32(&part[threadIdx.x]), r));
    (which == 0 ? a.kmean : a.vmean)[head * 64 + threadIdx.x] = s * a.scale;
  }
  cluster_sync();   // no block leaves while another may read its sums
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
  if (col < cols2)
    for (int b = g; b < n_blocks; b += 32) s += __ldcg(partials + static_cast<size_t>(b) * cols2 + col);
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

template <int PASSES>
cudaError_t launch_build(const Plan& pl, int grid, const void* K, const void* V, void* Kc, void* Vc, int64_t kc_rows,
                         int32_t* idx, float* partials, int do_mean, const int32_t* slot_of_token, uint32_t* status,
                         float* zero_kmean, float* zero_vmean, cudaStream_t st) {
  const size_t smem = do_mean ? static_cast<size_t>(kBuildWarps) * PASSES * 256 * sizeof(float) : 0;
  if (smem > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(build_kv_kernel<PASSES>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  return launch_dependent(build_kv_kernel<PASSES>, grid, kBuildThreads, smem, st, pl, static_cast<const uint4*>(K),
                          static_cast<const uint4*>(V), static_cast<uint4*>(Kc), static_cast<uint4*>(Vc), kc_rows, idx, partials,
                          do_mean, slot_of_token, status, zero_kmean, zero_vmean);
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

int build_passes(const Plan& pl) { return (pl.H * 8 + 31) / 32; }

int build_kv_blocks_per_sm(const Plan& pl) { return kBuildBlocks[build_passes(pl)]; }

int build_kv_grid(const Plan& pl, int sm_count) {
  const int64_t by_rows = (pl.n_tok + kBuildWarps - 1) / kBuildWarps;
  int64_t g = static_cast<int64_t>(sm_count) * build_kv_blocks_per_sm(pl);
  if (g > by_rows) g = by_rows;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

size_t build_kv_ws_bytes(const Plan& pl, int sm_count) {
  return static_cast<size_t>(build_kv_grid(pl, sm_count)) * 2 * pl.H * pl.d * sizeof(float);
}

cudaError_t launch_build_kv(const Plan& pl, int sm_count, const void* K, const void* V, void* Kc, void* Vc,
                            int32_t* idx, float* kmean, float* vmean, void* ws, cudaStream_t st,
                            const int32_t* caller_idx, int32_t* slot_of_token, int64_t kc_rows, bool sums_only,
                            void* clear_status) {
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
  const int grid = build_kv_grid(pl, sm_count);
  const int do_mean = (pl.mean_fill != 0 && pl.n_dropped > 0) ? 1 : 0;
  float* partials = static_cast<float*>(ws);
  uint32_t* status = static_cast<uint32_t*>(clear_status);
  const bool zero_mean = pl.mean_fill != 0 && !do_mean;
  float* zk = zero_mean ? kmean : nullptr;
  float* zv = zero_mean ? vmean : nullptr;
  const int passes = build_passes(pl);
  cudaError_t e;
  switch (passes) {
    case 1: e = launch_build<1>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 2: e = launch_build<2>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 3: e = launch_build<3>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 4: e = launch_build<4>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 5: e = launch_build<5>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 6: e = launch_build<6>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 7: e = launch_build<7>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    case 8: e = launch_build<8>(pl, grid, K, V, Kc, Vc, kc_rows, idx, partials, do_mean, slot_of_token, status, zk, zv, st); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess || !do_mean) return e;
  const int cols2 = 2 * pl.H * pl.d;
  const float inv_count = sums_only ? 1.0f : 1.0f / static_cast<float>(pl.n_dropped);
  return launch_dependent(mean_finalize_kernel, (cols2 + 31) / 32, 1024, 0, st, partials, grid, cols2, inv_count, kmean, vmean);
}

}  // namespace avggt
