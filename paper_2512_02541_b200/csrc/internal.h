// Declarations shared by the translation units of libavggt (not part of the ABI).
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "plan.h"

namespace avggt {

// ---- shared host helpers (api.cu)
struct DeviceInfo { int sm_count; int cc_major; };
// Properties of the current device.  AVGGT_OK only on an sm_100 device.
int device_info(DeviceInfo* out);
// Map a CUDA error to an AVGGT_* code, keeping its text for avggt_last_cuda_error.
int record_cuda(cudaError_t e);
// Keep `text` for avggt_last_cuda_error; returns AVGGT_ERR_CUDA.
int record_message(const char* text);
// The outcome of a launcher that encodes tensor maps.
inline int record_launch(cudaError_t e, bool tmap_failed) {
  return tmap_failed ? record_message("cuTensorMapEncodeTiled failed") : record_cuda(e);
}

// Launch of a kernel that may be scheduled, up to its grid_dependency_wait, while the kernel before it in the stream ends:
// the launch and the preparation of the layer's kernels (tensor memory, barriers) hide behind one another.
// cluster: thread blocks per cluster.
template <typename... P, typename... A>
cudaError_t launch_dependent_cluster(void (*kernel)(P...), unsigned grid, unsigned cluster, unsigned block, size_t smem, cudaStream_t st,
                                     const A&... args) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_dependent(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, const A&... args) {
  return launch_dependent_cluster(kernel, grid, 1, block, smem, st, args...);
}

constexpr size_t kAttnStatusBytes = 256;   // status block at the start of the attention workspace

// Clears the status block of a launch that no kernel of this library has cleared it for (global_attn.cu).
cudaError_t launch_clear_status(void* status, cudaStream_t st);

// ---- K/V compaction (build_kv.cu)
int build_kv_grid(const Plan& pl, int sm_count);
int build_kv_blocks_per_sm();
size_t build_kv_ws_bytes(const Plan& pl, int sm_count);
// What a call gets by with, on fewer blocks (above 16 heads a block per SM).
size_t build_kv_min_ws_bytes(const Plan& pl, int sm_count);
// caller_idx / slot_of_token: both null for the window rule of Sec. 4.3; for a caller-chosen retained set,
// the M retained token indices (device) and the [n_tok] map the call fills (device).
// kc_rows: rows per head of Kc / Vc (0 = M; larger when they are one rank's slot of an exchange buffer).
// sums_only: kmean / vmean receive the un-normalised sums over the dropped rows instead of the means.
// clear_status: the status block (kAttnStatusBytes) of the attention launch that follows in the stream, or null.
// Returns cudaSuccess, or an error; *tmap_failed is set when a tensor map could not be encoded.
cudaError_t launch_build_kv(const Plan& pl, int sm_count, const void* K, const void* V, void* Kc, void* Vc,
                            int32_t* idx, float* kmean, float* vmean, void* ws, size_t ws_bytes, cudaStream_t st, bool* tmap_failed,
                            const int32_t* caller_idx = nullptr, int32_t* slot_of_token = nullptr,
                            int64_t kc_rows = 0, bool sums_only = false, void* clear_status = nullptr);

// Frame-sharded layer: the ranks' slots of the exchange buffer -> one compact K/V pair, and the mean
// pair from the all-reduced sums.
constexpr int kMaxShardRanks = 64;
cudaError_t launch_assemble_shards(const void* gathered, int n_ranks, const int64_t* kept, int H, int d, int64_t slot_rows,
                                   void* Kc, void* Vc, const float* sums, int64_t n_dropped_total, float* kmean,
                                   float* vmean, cudaStream_t st);

// ---- attention (global_attn.cu)
size_t global_attn_ws_bytes(const Plan& pl, int sm_count);
// Returns cudaSuccess, or an error; *tmap_failed is set when a tensor map could not be encoded.
// slot_of_token: null for the window rule; else the map written by the indexed compaction.
// status_cleared: the compaction before it in the stream has cleared the status block.
cudaError_t launch_global_attn(const Plan& pl, int sm_count, const void* Q, const void* K, const void* V,
                               const void* Kc, const void* Vc, const float* kmean, const float* vmean, void* O,
                               float* lse, void* ws, cudaStream_t st, bool* tmap_failed,
                               const int32_t* slot_of_token = nullptr, bool status_cleared = false);

// Frame attention (Sec. 4.2): the same kernel, one independent dense problem per frame.
cudaError_t launch_frame_attn(const Plan& pl, int sm_count, const void* Q, const void* K, const void* V, void* O, float* lse,
                              void* ws, cudaStream_t st, bool* tmap_failed);

// ---- K/V projection with the compaction in its epilogue (project_kv.cu)
size_t project_kv_ws_bytes(const Plan& pl, int sm_count);
// X [n_tok, model_dim], Wk / Wv [H * d, model_dim] (the layout of a linear layer's weight), bias_k / bias_v [H * d] or
// null; K / V [n_tok, H, d] or null (written when given); the other outputs as for launch_build_kv.
cudaError_t launch_project_kv(const Plan& pl, int sm_count, int model_dim, const void* X, const void* Wk, const void* Wv,
                              const float* bias_k, const float* bias_v, void* K, void* V, void* Kc, void* Vc, int32_t* idx,
                              float* kmean, float* vmean, void* ws, cudaStream_t st, bool* tmap_failed);

}  // namespace avggt
