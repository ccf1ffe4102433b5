// Parameters and constants shared by the top-B kernels (bd_select.cu, bd_topk_long.cu).
#pragma once

#include "bd_common.cuh"

namespace bd {

constexpr int kTopkThreads = 1024;
constexpr int kBins = 4096;                   // linear histogram bins of the value range
constexpr int kBinCandMax = 2048;             // items of the boundary bin ranked exactly

struct TopkParams {
  const float* score;      // [units][n_mid_pad]
  int32_t* idx_out;        // [units][budget]
  int32_t* count_out;      // [units]
  int t_ctx, budget, n_sink, n_recent, chunk, n_mid_pad;
  int keep_all;            // budget >= t_ctx
  const int32_t* seq_lens; // per-sequence context lengths [batch] or null (all t_ctx)
  int h_kv;
  int* status;
};

// A unit whose context fits the budget keeps every position (the B >= T rule).  Executed by
// `n_threads` threads, tid of them this one.
__device__ __forceinline__ bool topk_keep_all(const TopkParams& p, int unit, int t_u, int32_t* out, int tid,
                                              int n_threads) {
  if (!p.keep_all && p.budget < t_u) return false;
  for (int i = tid; i < p.budget; i += n_threads) out[i] = i < t_u ? i : -1;
  if (tid == 0) p.count_out[unit] = t_u;
  return true;
}

// Selection for middles (or chunk counts) beyond the register-resident kernels of
// bd_select.cu, and the selections that rank nothing.
cudaError_t launch_topk_long(const TopkParams& p, int units, int n_items, cudaStream_t stream);
cudaError_t launch_topk_plain(const TopkParams& p, int units, cudaStream_t stream);

}  // namespace bd
