// What the two verify kernels (mma.sync: bd_verify.cu, tcgen05: bd_verify_tc.cu) share: the
// parameters, and the stream-K layout of the (unit, key tile) list.
#pragma once

#include "bd_common.cuh"

namespace bd {

constexpr int kVMaxSeg = 33;          // bound on the segments of one unit
constexpr int kVTcKeys = 128;         // keys per tile of verify_tc_kernel
constexpr int kVTcThreads = 320;      // its producer, MMA issuer and eight softmax warps

struct VerifyParams {
  const __nv_bfloat16* q;
  __nv_bfloat16* o;
  float* lse;
  float* o_part;       // [units][max_seg] partials of nq_rows x D floats: verify_kernel's [nq_rows][D],
                       // verify_tc_kernel's [D/4][nq_rows] float4
  float* lse_part;     // [units][max_seg][nq_rows]
  int* counters;       // [units]
  int* nseg;           // [units] segments of each unit (wide plans: read by verify_merge_kernel)
  int* status;
  const int32_t* seq_lens;  // per-sequence context lengths [batch] or null (all t_ctx)
  int h_kv;
  int n_q, nq_rows, t_ctx, tiles_per_unit, max_seg;
  // verify_tc_kernel: query rows of a (sequence, KV head) beyond what one CTA holds are cut into
  // row_chunks chunks of nq_rows rows (the last may hold fewer): a "unit" below is one
  // (sequence, KV head, chunk), and a KV head's chunks are adjacent in the unit list, so
  // CTAs streaming the same keys run side by side (the second read hits L2).
  int rows_total;      // group * n_q
  int row_chunks;
  int seg_cost;        // virtual tiles charged for each unit a CTA starts (see verify_plan)
  int vtiles_per_cta;  // contiguous range of the virtual tile list per CTA
  float scale_log2;    // log2(e) / sqrt(D)
  int units;           // batch * h_kv * row_chunks
  int tile_rows;       // query rows of the first M tile of a chunk (verify_tc_kernel)
};

// The global tile list is cut into equal CTA ranges after every unit's tiles are preceded
// by `seg_cost` virtual tiles: a CTA whose range starts a unit (and so stops to merge one
// segment and load new queries) receives that many fewer real tiles.
// The CTA whose range holds real tile g.
__host__ __device__ __forceinline__ int tile_owner(int g, int tpu, int a, int vtpc) {
  const int u = g / tpu;
  return (u * (tpu + a) + a + (g - u * tpu)) / vtpc;
}

// The same layout seen per unit: unit u spans virtual tiles [vbase(u), vbase(u + 1)), its
// `a` virtual tiles first, then its real tiles 0 .. tiles(u) - 1; the list is cut into
// ranges of vtpc virtual tiles, one per CTA.  pref (shared memory, per-sequence lengths)
// holds vbase(u) for u = 0 .. units; null means every unit has tpu real tiles.
struct VerifyMap {
  const int* pref;
  int tpu, a, units, vtpc;
  __device__ __forceinline__ int vbase(int u) const { return pref ? pref[u] : u * (tpu + a); }
  __device__ __forceinline__ int tiles(int u) const { return vbase(u + 1) - vbase(u) - a; }
  __device__ __forceinline__ int unit_of(int v) const {   // the unit whose span holds v
    if (!pref) return v / (tpu + a);
    int lo = 0, hi = units - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (pref[mid] <= v) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  }
  // real tiles of unit u inside the virtual range [v0, v1)
  __device__ __forceinline__ int first_tile(int u, int v0) const { return max(0, v0 - vbase(u) - a); }
  __device__ __forceinline__ int end_tile(int u, int v1) const { return min(tiles(u), v1 - vbase(u) - a); }
  __device__ __forceinline__ int owner(int u, int tile) const { return (vbase(u) + a + tile) / vtpc; }
};

// Per-sequence lengths: every CTA lays out the units' virtual tile spans itself, pref[u] =
// vbase(u) for u = 0 .. units, by all NTHREADS threads (wtot: one int per warp).  The lengths
// may come from the preceding kernel, so the caller has passed the dependency wait.
template <int NTHREADS, int KEYS>
__device__ __forceinline__ void lay_out_units(const VerifyParams& p, int n_units, int* wtot, int* pref) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int per = (n_units + NTHREADS - 1) / NTHREADS;
  const int u0 = min(n_units, tid * per), u1 = min(n_units, u0 + per);
  auto span = [&](int u) {
    const int t_u = unit_context(p.seq_lens, u / p.row_chunks, p.h_kv, p.t_ctx, nullptr);
    return (t_u + p.n_q + KEYS - 1) / KEYS + p.seg_cost;
  };
  int sum = 0;
  for (int u = u0; u < u1; ++u) sum += span(u);
  int incl = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += y;
  }
  if (lane == 31) wtot[warp] = incl;
  __syncthreads();
  int run = incl - sum;
  for (int w = 0; w < warp; ++w) run += wtot[w];
  for (int u = u0; u < u1; ++u) {
    pref[u] = run;
    run += span(u);
  }
  if (tid == NTHREADS - 1) pref[n_units] = run;
  __syncthreads();
}

// The tcgen05 kernel's instance for q_tiles (1 or 2) M tiles of query rows per unit, and its
// shared memory without the units' table of per-sequence lengths.
size_t verify_tc_smem(int head_dim, int q_tiles);
const void* verify_tc_fn(int head_dim, int q_tiles, bool ragged);
cudaError_t launch_verify_tc_merge(int head_dim, int units, const VerifyParams& p, cudaStream_t stream);

}  // namespace bd
