// Verifier block attention (Algorithm 2, Verify): n_q queries per head at positions
// t_ctx .. t_ctx+n_q-1 over keys [0, t_ctx + i] (causal inside the block), up to 24 query rows per
// KV head (more run on verify_tc_kernel, bd_verify_tc.cu); the plan and the launch of both.
//
// Persistent, stream-K scheduled: the (unit, 64-key tile) pairs of all (sequence, KV head)
// units form one list that is cut into contiguous ranges, one per CTA, of equal cost: each
// unit's tiles are preceded by a few virtual tiles that stand for the cost of starting a
// unit, so every SM streams about the same time whatever the batch.  A range covers one or
// two units; each piece of a unit ("segment") ends in a normalised partial (o, lse), and
// the last CTA to finish a unit merges its segments (log-sum-exp) into the final bf16
// output, staging the partials in shared memory with cp.async (one round trip).
//   warp 4      TMA producer: 64-key K and V tiles, 128-byte swizzle, 5-stage ring,
//               streaming straight across segment boundaries.  Context rows [0, t_ctx)
//               are streamed before the grid-dependency wait (they are not written by
//               the preceding kernel); the wait comes before the first tile that holds
//               the block's own rows (before the first load when per-sequence lengths
//               are given: any tile may then hold some sequence's block rows);
//   warps 0..3  consumers on mma.sync (bd_attn_warp.cuh): the GQA group's packed query
//               rows are the N side of S^T = K Q^T.
#include <algorithm>
#include <climits>

#include "bd_attn_warp.cuh"
#include "bd_common.cuh"
#include "bd_internal.h"
#include "bd_verify.cuh"

namespace bd {

constexpr int kVKeys = 64;            // keys per pipeline stage
constexpr int kVConsumers = 4;        // consumer warps
constexpr int kVThreads = 160;        // + one producer warp
constexpr int kVStages = 5;
// Most query rows of a KV head that verify_kernel takes: three n8 tiles, up to which it streams at
// memory speed and starts sooner; with more, every tile of keys costs another pass of mma.sync
// and verify_tc_kernel is faster.  64 units of 16K, both sides measured: 28 rows 154.5 us here, 85.4
// there; 84 rows 313.8 / 89.1.  8 units of 4K: 24 rows 10.5 / 11.2, 36 rows 13.4 / 12.6, 84 rows 19.2 / 13.4.
constexpr int kVMaxRows = 24;
constexpr int kVTcRows = 16;          // query rows from which a large batch moves already
constexpr int kVTcMaxRows = 256;      // query rows of one unit of verify_tc_kernel: two M tiles
constexpr int kVMaxChunks = 3;        // row chunks of one (sequence, KV head): 768 query rows in all

template <int D, int NT>
struct VerifySmem {
  static constexpr int WK = kVConsumers;
  static constexpr int NQC = 8 * NT;
  static constexpr uint32_t TILE_BYTES = kVKeys * D * 2;
  static constexpr uint32_t STAGE_BYTES = 2 * TILE_BYTES;
  static constexpr size_t kStages = (size_t)kVStages * STAGE_BYTES;
  static constexpr size_t kMerge = (size_t)(3 * WK * NQC) * 4 + (size_t)WK * NQC * (D + 4) * 4;
  static constexpr size_t kWeights = (size_t)kVMaxSeg * NQC * 4;
  // layout after the 1 KB barrier block: stages | merge scratch | merge weights
  static constexpr size_t kTotal = 1024 + 1024 + kStages + kMerge + kWeights;
};

// WIDE: the instance for plans whose units span more CTAs than the last one can merge in a
// single staged round trip (small and mid-size batches).  Every CTA only writes its
// segment's partial, the unit's first CTA its segment count, and verify_merge_kernel,
// launched right after, merges them with the whole GPU: a last-CTA merge of ten to twenty
// parts cost 10-16 us at the end of the kernel.  A separate instance, so that the common
// case's code (and register allocation) stays as it is.
// NT: n8 tiles of query rows; SUBS: 16-key sub-tiles of a tile per consumer warp.
// UNIFORM: one shared context length; the other instances lay out per-sequence lengths.
template <int D, int NT, int SUBS, bool UNIFORM, bool WIDE>
__global__ void __launch_bounds__(kVThreads, D == 128 && NT == 1 ? 1 : 0) verify_kernel(const VerifyParams p,
                                                           const __grid_constant__ CUtensorMap kmap,
                                                           const __grid_constant__ CUtensorMap vmap) {
  using L = VerifySmem<D, NT>;
  constexpr int WK = L::WK, NQC = L::NQC;
  constexpr uint32_t HALF_BYTES = kVKeys * 128;
  constexpr int STAGES = kVStages;
  static_assert(16 * SUBS * kVConsumers == kVKeys, "the warps' sub-tiles make up a tile");

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty_bar = full_bar + STAGES;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(empty_bar + STAGES);
  int* last_flag = const_cast<int*>(abort_flag) + 1;
  uint8_t* stage_base = smem + 1024;
  float* m_s = reinterpret_cast<float*>(stage_base + L::kStages);
  float* l_s = m_s + WK * NQC;
  float* f_s = l_s + WK * NQC;
  float* o_s = f_s + WK * NQC;
  float* w_s = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(m_s) + L::kMerge);
  int* pref = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(w_s) + L::kWeights);   // ragged: [units + 1]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_units = p.units;
  VerifyMap map{nullptr, p.tiles_per_unit, p.seg_cost, n_units, p.vtiles_per_cta};
  if (!UNIFORM) {
    // per-sequence lengths: every CTA lays out the units' virtual tile spans itself (the
    // lengths may come from the preceding kernel, so after the dependency wait)
    grid_dependency_wait();
    lay_out_units<kVThreads, kVKeys>(p, n_units, reinterpret_cast<int*>(smem + 512), pref);
    map.pref = pref;
    map.vtpc = max((pref[n_units] + (int)gridDim.x - 1) / (int)gridDim.x, p.vtiles_per_cta);
  }
  const int v_total = map.vbase(n_units);
  const int v0 = min(v_total, (int)blockIdx.x * map.vtpc), v1 = min(v_total, v0 + map.vtpc);
  if (v0 >= v1) return;                           // whole CTA idle
  const int u_first = map.unit_of(v0), u_last = map.unit_of(v1 - 1);
  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], kVConsumers);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();

  if (warp == kVConsumers) {
    // ------------------------------------------------------------------ producer
    allow_dependent_launch();
    if (lane == 0) {
      tma_prefetch_map(&kmap);
      tma_prefetch_map(&vmap);
      int issued = 0;
      // with per-sequence lengths any tile may hold some sequence's block rows (written by
      // the preceding kernels): the wait above came before the first load
      bool waited = !UNIFORM;
      bool stop = false;
      for (int unit = u_first; unit <= u_last && !stop; ++unit) {
        const int tb = map.first_tile(unit, v0), te = map.end_tile(unit, v1);
        for (int tile = tb; tile < te; ++tile) {
          const int t = issued;
          const int s = t % STAGES;
          if (t >= STAGES && !mbar_wait(&empty_bar[s], ((t / STAGES) & 1) ^ 1, p.status, abort_flag)) {
            stop = true;
            break;
          }
          const int key0 = tile * kVKeys;
          if (!waited && key0 + kVKeys > p.t_ctx) {    // this tile holds rows of the block itself
            grid_dependency_wait();
            waited = true;
          }
          uint8_t* st = stage_base + s * L::STAGE_BYTES;
          mbar_arrive_expect_tx(&full_bar[s], L::STAGE_BYTES);
#pragma unroll
          for (int h = 0; h < D / 64; ++h) tma_load_3d(st + h * HALF_BYTES, &kmap, &full_bar[s], 64 * h, key0, unit);
#pragma unroll
          for (int h = 0; h < D / 64; ++h)
            tma_load_3d(st + L::TILE_BYTES + h * HALF_BYTES, &vmap, &full_bar[s], 64 * h, key0, unit);
          issued = t + 1;
        }
      }
      if (*abort_flag) {   // never leave a copy in flight behind an aborted CTA
        for (int t = max(0, issued - STAGES); t < issued; ++t)
          mbar_wait(&full_bar[t % STAGES], (t / STAGES) & 1, p.status, nullptr);
      }
    }
    return;
  }

  // -------------------------------------------------------------------- consumers
  if (UNIFORM)   // the first unit's queries on their way into L2 while the predecessor finishes
    prefetch_lines_l2(p.q + (size_t)u_first * p.nq_rows * D, (size_t)p.nq_rows * D * 2, tid, kVConsumers * 32);
  grid_dependency_wait();                        // the queries come from the preceding kernels
  allow_dependent_launch();
  const int tig = lane & 3;
  const int nq = p.nq_rows;                      // query rows of a unit
  constexpr int NCT = kVConsumers * 32;          // consumer threads
  int lim[NT][2];                                // last visible key of each of this thread's columns

  bool alive = true;   // false once this warp's wait gave up (the abort flag is then set)
  int t = 0;
  // the next unit of this range with real tiles here (past u_last: none)
  auto next_unit = [&](int u) {
    while (u <= u_last && map.first_tile(u, v0) >= map.end_tile(u, v1)) ++u;
    return u;
  };
  auto unit_q = [&](int u, uint32_t (&bq)[NT][D / 16][2]) {
    WarpAttn<D, NT>::load_q(bq, p.q + (size_t)u * nq * D, nq, 0, lane);
  };
  uint32_t bq[NT][D / 16][2];
  int unit = next_unit(u_first);
  if (unit <= u_last) unit_q(unit, bq);
  for (; unit <= u_last;) {
    const int tb = map.first_tile(unit, v0), te = map.end_tile(unit, v1);
    const size_t row0 = (size_t)unit * nq;       // its first row in q / o / lse
    const int t_unit =
        UNIFORM ? p.t_ctx : unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 ? p.status : nullptr);
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int col = 8 * nt + 2 * tig + e;
        lim[nt][e] = col < nq ? t_unit + col % p.n_q : -1;
      }
    WarpAttn<D, NT> wa;
    wa.init();
    for (int tile = tb; tile < te && alive; ++tile, ++t) {
      const int s = t % STAGES;
      if (!mbar_wait(&full_bar[s], (t / STAGES) & 1, p.status, abort_flag)) {
        alive = false;
        break;
      }
      const uint32_t kbase = smem_u32(stage_base + s * L::STAGE_BYTES);
      const uint32_t vbase = kbase + L::TILE_BYTES;
#pragma unroll
      for (int sub = 0; sub < SUBS; ++sub) {
        const int kb = 16 * (warp + kVConsumers * sub);
        const int key_base = tile * kVKeys + kb;
        // (a shorter sequence's last tile reaches cache rows past its own block, which nobody has promised to
        // be finite; past the longest block the tensor map reads zeros)
        wa.step(kbase, vbase, HALF_BYTES, kb, bq, p.scale_log2, lane,
                [&](int ko, int nt, int e) { return key_base + ko <= lim[nt][e]; },
                UNIFORM ? INT_MAX : t_unit + p.n_q - 1 - tile * kVKeys);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_bar[s]);
    }
    // the next unit's queries are requested now, so that they arrive while this segment
    // closes (its merge, partial write and arrival take several round trips to memory)
    const int next = next_unit(unit + 1);
    if (next <= u_last && alive) unit_q(next, bq);
    wa.finish_rows();

    // ---------------------------------------------------------------- end of a segment
    wa.store(m_s, l_s, o_s, warp, NQC, 0, lane);
    named_bar(1, NCT);
    const int c = blockIdx.x;
    const int c_first = map.owner(unit, 0);
    const int c_last = map.owner(unit, map.tiles(unit) - 1);
    const int n_seg = c_last - c_first + 1;
    if (WIDE && c == c_first && tid == 0) p.nseg[unit] = n_seg;
    if (n_seg == 1) {
      merge_warps_and_store<D, WK>(m_s, l_s, f_s, o_s, NQC, nq, p.lse ? p.lse + row0 : nullptr,
                                           static_cast<void*>(p.o + row0 * D), true, tid, NCT, 1);
    } else if constexpr (WIDE) {
      const size_t slot = (size_t)unit * p.max_seg + (c - c_first);
      merge_warps_and_store<D, WK>(m_s, l_s, f_s, o_s, NQC, nq, p.lse_part + slot * nq,
                                           static_cast<void*>(p.o_part + slot * nq * D), false,
                                           tid, NCT, 1);
    } else {
      const size_t slot = (size_t)unit * p.max_seg + (c - c_first);
      merge_warps_and_store<D, WK>(m_s, l_s, f_s, o_s, NQC, nq, p.lse_part + slot * nq,
                                           static_cast<void*>(p.o_part + slot * nq * D), false,
                                           tid, NCT, 1);
      __threadfence();
      named_bar(1, NCT);
      if (tid == 0) *last_flag = (atomicAdd(&p.counters[unit], 1) == n_seg - 1);
      named_bar(1, NCT);
      if (*last_flag) {
        __threadfence();
        const size_t base = (size_t)unit * p.max_seg;
        merge_partials<D>(p.o_part + base * nq * D, p.lse_part + base * nq, n_seg, nq, (size_t)nq * D, (size_t)nq,
                          p.o + row0 * D, p.lse ? p.lse + row0 : nullptr, [](int r) { return r; },
                          w_s, tid, NCT, 1, m_s, L::kMerge / 4);
        if (tid == 0) p.counters[unit] = 0;
      }
    }
    named_bar(1, NCT);                           // scratch free for the next segment
    // every consumer warp takes the same decision to stop after a timed-out wait
    if (tid == 0) last_flag[1] = *abort_flag;
    named_bar(1, NCT);
    if (last_flag[1]) break;
    unit = next;
  }
}

// Merge of the segments' partials for the wide plans: one CTA per (unit, output row); a
// unit whose segment count is 1 was written by the verify kernel itself.  Thread t takes
// four adjacent columns (t % (D/4)) of the segments s = t / (D/4) (mod 128 / (D/4)), so
// every part of the row is requested at once: the lse values, then the rows, two round
// trips to L2 in all; the groups' sums meet in shared memory.
template <int D>
__global__ void __launch_bounds__(128) verify_merge_kernel(const float* o_part, const float* lse_part,
                                                           const int* nseg, int max_seg, int nq, __nv_bfloat16* o,
                                                           float* lse) {
  constexpr int Q = D / 4;                 // column quads per row
  constexpr int NG = 128 / Q;              // segment groups
  constexpr int PER = (kVMaxSeg + NG - 1) / NG;
  grid_dependency_wait();
  allow_dependent_launch();
  __shared__ float w[kVMaxSeg];
  __shared__ float4 part[NG][Q];
  const int unit = blockIdx.x, r = blockIdx.y, tid = threadIdx.x;
  const int n = min(__ldcg(nseg + unit), kVMaxSeg);
  if (n <= 1) return;
  const size_t orow = (size_t)unit * nq + r;        // the output row
  const size_t base = (size_t)unit * max_seg;
  if (tid < 32) {
    const float l0 = tid < n ? __ldcg(lse_part + (base + tid) * nq + r) : -INFINITY;
    const float l1 = tid + 32 < n ? __ldcg(lse_part + (base + tid + 32) * nq + r) : -INFINITY;
    float mx = fmaxf(l0, l1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float e0 = mx == -INFINITY ? 0.f : fast_exp2((l0 - mx) * kLog2e);
    const float e1 = mx == -INFINITY ? 0.f : fast_exp2((l1 - mx) * kLog2e);
    float tot = e0 + e1;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, off);
    const float inv = tot > 0.f ? 1.f / tot : 0.f;
    if (tid < n) w[tid] = e0 * inv;
    if (tid + 32 < n) w[tid + 32] = e1 * inv;
    if (tid == 0 && lse) lse[orow] = mx == -INFINITY ? -INFINITY : mx + logf(tot);
  }
  const int q = tid % Q, g = tid / Q;
  float4 v[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int sg = g + NG * k;
    v[k] = sg < n ? __ldcg(reinterpret_cast<const float4*>(o_part + ((base + sg) * nq + r) * D) + q)
                  : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __syncthreads();                                  // the weights
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int sg = g + NG * k;
    const float wk = sg < n ? w[sg] : 0.f;
    if (wk != 0.f) {                                // an empty part never enters the sum
      acc.x += wk * v[k].x;
      acc.y += wk * v[k].y;
      acc.z += wk * v[k].z;
      acc.w += wk * v[k].w;
    }
  }
  part[g][q] = acc;
  __syncthreads();
  if (g == 0) {
#pragma unroll
    for (int h = 1; h < NG; ++h) {
      const float4 b = part[h][q];
      acc.x += b.x;
      acc.y += b.y;
      acc.z += b.z;
      acc.w += b.w;
    }
    uint2 packed;
    packed.x = pack_bf16x2(acc.x, acc.y);
    packed.y = pack_bf16x2(acc.z, acc.w);
    *reinterpret_cast<uint2*>(o + orow * D + 4 * q) = packed;
  }
}

// ============================================================================ host side

namespace {

struct KernelInfo {
  void* fn;
  size_t smem;
  size_t merge_floats;   // the staging area a unit's last CTA merges the segments' partials in
};

template <int D, int NT, bool UNIFORM, bool WIDE>
KernelInfo info() {
  return {reinterpret_cast<void*>(&verify_kernel<D, NT, kVKeys / (16 * kVConsumers), UNIFORM, WIDE>), VerifySmem<D, NT>::kTotal,
          VerifySmem<D, NT>::kMerge / 4};
}

KernelInfo select_kernel(int d, int nt, bool uniform, bool wide) {
#define BD_VK(DD, N, U)                     \
  if (d == DD && nt == N && uniform == U) \
    return wide ? info<DD, N, U, true>() : info<DD, N, U, false>();
  BD_VK(64, 1, true) BD_VK(64, 3, true) BD_VK(64, 1, false) BD_VK(64, 3, false)
  BD_VK(128, 1, true) BD_VK(128, 3, true) BD_VK(128, 1, false) BD_VK(128, 3, false)
#undef BD_VK
  return {nullptr, 0, 0};
}

// Resident CTAs per SM of a kernel (cached per kernel and device).
int occupancy(const KernelInfo& k) {
  static thread_local void* last_fn = nullptr;
  static thread_local int last_dev = -1, last_occ = 1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (k.fn == last_fn && dev == last_dev) return last_occ;
  int occ = 1;
  if (allow_shared_memory(k.fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k.fn, kVThreads, k.smem) != cudaSuccess || occ < 1)
    occ = 1;
  (void)cudaGetLastError();
  last_fn = k.fn;
  last_dev = dev;
  last_occ = occ;
  return occ;
}

}  // namespace

// Blocks that verify_kernel could take but verify_tc_kernel streams faster: a third n8 tile slows
// every tile of keys in the one (8 rows 81.5 us, 24 rows 86.3 us for 64 units of 16K), while the other
// costs the same up to 128 rows and wants a merge launch, which pays once the batch fills the SMs by itself.
// verify_kernel / verify_tc_kernel, d 128, us: 64 units, 24 rows, of 1K 17.1 / 15.9, 4K 31.2 / 29.3, 16K 86.5 / 85.2;
// 128 units, 21 rows, of 4K 50.1 / 48.2, 16K 159.3 / 158.3; 12 rows: 15.0 / 16.3, 29.8 / 29.9, 85.3 / 85.3; 32 units, 24
// rows, of 16K 47.9 / 49.4; d 64, 64 units of 16K 49.8 / 58.5; per-sequence lengths, 21 rows 48.2 / 48.4.  Three full
// n8 tiles over more than a million keys in many units stay: 24 rows, 128 units of 16K 158.2 / 159.7, 160 of 8K 104.7 /
// 105.3, 256 of 8K 159.5 / 161.4 (but 128 of 8K 86.5 / 85.8, 256 of 4K 88.1 / 87.6, 96 of 16K 122.2 / 121.9).
static bool tc_streams_better(const bd_shape& s, int n_q) {
  const long units = (long)s.batch * s.h_kv, keys = (long)s.t_ctx + n_q;
  if (s.head_dim != 128 || s.seq_lens != nullptr || 3 * units <= current_sm_count() || keys < 1024) return false;
  return s.h_q / s.h_kv * n_q <= 21 || units < 128 || units * keys < 5L << 18;
}

// What a block's plan depends on beside its row count: the kernel (and its instance), the chunks, the tiles.
struct VerifyRoute {
  long rows;            // group * n_q
  bool tc;              // verify_tc_kernel
  int nt, chunks, tiles;
  bool operator==(const VerifyRoute& o) const { return tc == o.tc && nt == o.nt && chunks == o.chunks && tiles == o.tiles; }
};
static VerifyRoute verify_route(const bd_shape& s, int n_q) {
  VerifyRoute r;
  r.rows = (long)(s.h_q / s.h_kv) * n_q;
  r.tc = r.rows > kVMaxRows || (r.rows > kVTcRows && tc_streams_better(s, n_q));
  // more query rows than one CTA holds: chunks of equal size
  r.chunks = r.tc ? (int)((r.rows + kVTcMaxRows - 1) / kVTcMaxRows) : 1;
  r.nt = r.tc ? 0 : r.rows <= 8 ? 1 : 3;
  const int keys = r.tc ? kVTcKeys : kVKeys;
  r.tiles = (int)(((long)s.t_ctx + n_q + keys - 1) / keys);
  return r;
}

bool verify_plan(const bd_shape& s, int n_q, VerifyPlan* plan) {
  const VerifyRoute route = verify_route(s, n_q);
  const bool ragged = s.seq_lens != nullptr, tc = route.tc;
  const long rows_total = route.rows;
  const int chunks = route.chunks, nt = route.nt;
  if (chunks > kVMaxChunks) return false;
  const int nq_rows = (int)((rows_total + chunks - 1) / chunks);
  const int q_tiles = tc ? (nq_rows > 128 ? 2 : 1) : 0;
  KernelInfo k = {nullptr, 0, 0};
  if (!tc) {
    k = select_kernel(s.head_dim, nt, !ragged, false);
    if (!k.fn) return false;
  }
  const int keys = tc ? kVTcKeys : kVKeys;
  plan->nq_rows = nq_rows;
  plan->rows_total = (int)rows_total;
  plan->row_chunks = chunks;
  plan->q_tiles = q_tiles;
  plan->nt = nt;
  plan->smem_bytes = tc ? verify_tc_smem(s.head_dim, q_tiles) : k.smem;
  plan->tiles_per_unit = route.tiles;
  const long units = (long)s.batch * s.h_kv * chunks;
  const int tpu = plan->tiles_per_unit;
  const long ctas = std::max(1, current_sm_count() * (tc ? 1 : occupancy(k)));
  // A unit boundary inside a CTA's range (the segment's merge of the warps' partials, its
  // write, the arrival, the merge by the unit's last CTA) costs about 5 us of streaming time;
  // charge it as virtual tiles at the rate one CTA streams at when every SM streams
  // (~6.5 TB/s over all SMs).  Traced: with 3 us charged, the CTAs holding a boundary ended
  // their last tile ~5 us after the others; swept at 1-12 us, 5 us gave the shortest step.
  const double tile_bytes = (double)keys * s.head_dim * 2 * 2;
  const double tile_us = tile_bytes / (6.5e6 / (double)std::max(1, current_sm_count()));
  const int a = (int)std::min(16.0, std::max(0.0, 5.0 / tile_us + 0.5));
  const long vtotal = units * (tpu + a);
  if (vtotal >= (1L << 31)) return false;
  long vtpc = (vtotal + ctas - 1) / ctas;
  vtpc = std::max<long>(vtpc, (tpu + a + kVMaxSeg - 2) / (kVMaxSeg - 1));   // <= kVMaxSeg segments
  plan->seg_cost = a;
  plan->tiles_per_cta = (int)vtpc;
  plan->grid = (int)((vtotal + vtpc - 1) / vtpc);
  int max_seg = 1;
  for (long u = 0; u < std::min(units, vtpc); ++u) {   // (units' offsets in the CTA ranges repeat after vtpc units)
    const int c0 = tile_owner((int)(u * tpu), tpu, a, (int)vtpc);
    const int c1 = tile_owner((int)(u * tpu + tpu - 1), tpu, a, (int)vtpc);
    max_seg = std::max(max_seg, c1 - c0 + 1);
  }
  if (max_seg > kVMaxSeg) return false;
  plan->max_seg = max_seg;
  if (ragged) {
    // per-sequence lengths: the kernel cuts the ranges itself over the actual tiles, no
    // shorter than the bound that keeps every unit within kVMaxSeg segments; the units'
    // span table takes (units + 1) ints of shared memory
    plan->tiles_per_cta = (int)((tpu + a + kVMaxSeg - 2) / (kVMaxSeg - 1));
    plan->max_seg = kVMaxSeg;
    plan->smem_bytes += align_up((size_t)(units + 1) * 4, 16);
    if (plan->smem_bytes > 227 * 1024) return false;
  }
  // the unit's last CTA merges its segments in one staged round trip while they fit its
  // merge area; more segments take the chunked merge of the wide instance
  plan->wide = tc ? plan->max_seg > 1 : (size_t)plan->max_seg * nq_rows * s.head_dim > k.merge_floats;
  return true;
}

size_t verify_partials_bytes(const bd_shape& s, const VerifyPlan& plan) {
  if (plan.max_seg <= 1) return 0;
  const size_t units = (size_t)s.batch * s.h_kv * plan.row_chunks;
  const size_t rows = units * plan.max_seg * plan.nq_rows;
  return align_up(rows * s.head_dim * 4, 256) + align_up(rows * 4, 256) + (plan.wide ? align_up(units * 4, 256) : 0);
}

size_t verify_region_bytes(const bd_shape& s, int n_q) {
  size_t bytes = 0;
  for (int n = 1; n <= n_q; ++n) {
    if (n < n_q && verify_route(s, n) == verify_route(s, n + 1)) continue;   // the longer one needs as much
    VerifyPlan vp;
    if (verify_plan(s, n, &vp)) bytes = std::max(bytes, verify_partials_bytes(s, vp));
  }
  return bytes;
}

cudaError_t launch_verify(const bd_shape& s, const VerifyPlan& plan, int n_q, const void* q,
                          const void* k_cache, const void* v_cache, void* o_out, float* lse_out,
                          void* ws_region, int* counters, int* status, cudaStream_t stream) {
  const int units = s.batch * s.h_kv;
  const int keys = plan.q_tiles ? kVTcKeys : kVKeys;
  CUtensorMap kmap, vmap;
  cudaError_t err = make_cache_map(&kmap, k_cache, units, s.t_cap, s.t_ctx + n_q, s.head_dim, keys);
  if (err != cudaSuccess) return err;
  err = make_cache_map(&vmap, v_cache, units, s.t_cap, s.t_ctx + n_q, s.head_dim, keys);
  if (err != cudaSuccess) return err;
  VerifyParams p;
  p.q = static_cast<const __nv_bfloat16*>(q);
  p.o = static_cast<__nv_bfloat16*>(o_out);
  p.lse = lse_out;
  const size_t rows = (size_t)units * plan.row_chunks * plan.max_seg * plan.nq_rows;
  p.o_part = static_cast<float*>(ws_region);
  p.lse_part = reinterpret_cast<float*>(static_cast<uint8_t*>(ws_region) + align_up(rows * s.head_dim * 4, 256));
  p.counters = counters;
  p.nseg = reinterpret_cast<int*>(reinterpret_cast<uint8_t*>(p.lse_part) + align_up(rows * 4, 256));
  p.status = status;
  p.n_q = n_q;
  p.nq_rows = plan.nq_rows;
  p.rows_total = plan.rows_total;
  p.row_chunks = plan.row_chunks;
  p.t_ctx = s.t_ctx;
  p.seq_lens = s.seq_lens;
  p.h_kv = s.h_kv;
  p.tiles_per_unit = plan.tiles_per_unit;
  p.seg_cost = plan.seg_cost;
  p.vtiles_per_cta = plan.tiles_per_cta;
  p.max_seg = plan.max_seg;
  p.scale_log2 = kLog2e / sqrtf((float)s.head_dim);
  p.units = units * plan.row_chunks;
  p.tile_rows = plan.q_tiles == 2 ? (plan.nq_rows + 1) / 2 : plan.nq_rows;
  const void* fn = plan.q_tiles ? verify_tc_fn(s.head_dim, plan.q_tiles, s.seq_lens != nullptr)
                                : select_kernel(s.head_dim, plan.nt, s.seq_lens == nullptr, plan.wide).fn;
  err = allow_shared_memory(fn);
  if (err != cudaSuccess) return err;
  CUtensorMap qmap;
  if (plan.q_tiles) {
    err = make_rows_map(&qmap, q, (long long)units * plan.rows_total, s.head_dim, 128);
    if (err != cudaSuccess) return err;
  }
  void* args[] = {&p, &kmap, &vmap, &qmap};   // (verify_kernel takes the first three)
  err = launch_kernel(fn, dim3(plan.grid), dim3(plan.q_tiles ? kVTcThreads : kVThreads), plan.smem_bytes, stream, args, 0);
  if (err != cudaSuccess || !plan.wide) return err;
  if (plan.q_tiles) return launch_verify_tc_merge(s.head_dim, p.units, p, stream);
  const float* op = p.o_part;
  const float* lp = p.lse_part;
  const int* ns = p.nseg;
  int max_seg = plan.max_seg, nq = plan.nq_rows;
  __nv_bfloat16* o = p.o;
  float* l = p.lse;
  void* margs[] = {&op, &lp, &ns, &max_seg, &nq, &o, &l};
  void* mfn = s.head_dim == 64 ? reinterpret_cast<void*>(&verify_merge_kernel<64>)
                               : reinterpret_cast<void*>(&verify_merge_kernel<128>);
  return launch_kernel(mfn, dim3(units, plan.nq_rows), dim3(128), 0, stream, margs, 0);
}

}  // namespace bd
