// KV-budget selection (Sec. 3.4 TopKChunks; Algorithm 2, sparsify) in two kernels (three
// in self mode, where window_lse_kernel first computes the window rows' normalisers, see
// its own comment below):
//
// score_kernel  (tcgen05)  score[k] = sum_{h in group, w < W, k <= p_w} exp2(s_{h,w,k} log2e/sqrt(d)
//               - lse_{h,w} log2e) for every middle key k.  Keys sit on the M side of the
//               UMMA (128 keys per tile = the 128 TMEM lanes) and the group's window query
//               rows on N, so every epilogue thread owns one key and reduces its own TMEM
//               row: no cross-thread reduction.  Persistent CTAs (one per SM):
//                 warp 0   producer: K tiles by TMA (128-byte swizzle, 4-stage ring) and the
//                          unit's window queries into a double-buffered swizzled Q tile;
//                          the first stages' K tiles (context rows) stream before the
//                          grid-dependency wait, the queries (which bd_advance may have
//                          just rewritten) and the later tiles after it;
//                 warp 1   one lane issues tcgen05.mma into four fp32 TMEM accumulators
//                          (two when the window rows need more columns) and commits to
//                          the smem/TMEM barriers;
//                 warps 2-17 epilogue (four groups of 4, every fourth tile): tcgen05.ld,
//                          packed f32x2 FMA, ex2 (MUFU), packed row sums, coalesced store.
// top-B         one CTA per (sequence, KV head): a linear histogram between the min and
//               max score finds the bin holding the k-th largest; that bin's few items are
//               ranked exactly by (score desc, position asc) (4-pass radix select on the
//               fp32 bits when the bin is crowded); then an ascending compaction (warp
//               ballots + block scan) with sinks and recents.  topk_rows_kernel (token level)
//               and topk_rows_chunk_kernel (chunk level) here hold every item of a middle of up
//               to 16K positions in registers, topk_token_kernel up to 32K in shared memory;
//               bd_topk_long.cu spreads longer middles over a cluster.
#include <algorithm>
#include <climits>

#include "bd_common.cuh"
#include "bd_internal.h"
#include "bd_topk.cuh"

namespace bd {

constexpr int kSKeys = 128;          // keys per tile (UMMA M)
constexpr int kSThreads = 576;       // producer, MMA, 4 x 4 epilogue warps
constexpr int kSGroups = 4;          // epilogue groups of four warps
constexpr int kSQOffset = 12288;     // shared-memory offset of the window-query tiles

struct ScoreParams {
  const __nv_bfloat16* q_win;   // [units * nq_rows][D]
  const float* lse_win;         // [units * nq_rows] natural log
  float* score;                 // [units][n_mid_pad]
  int* status;
  int nq_rows, nq_pad, window, t_ctx, n_sink, mid_end, n_mid_pad;
  int tiles_per_unit, total_tiles, tiles_per_cta;
  int acc_stride;               // TMEM columns between accumulators
  int n_acc;                    // accumulators: tile i uses i % n_acc; epilogue group i % 4
  uint32_t tmem_cols;
  float scale_log2;
  const int32_t* seq_lens;      // per-sequence context lengths [batch] or null (all t_ctx)
  int h_kv;
  int window_ready;             // BD_SELECT_WINDOW_READY: the queries may load before the dependency wait
};

// RAGGED: per-sequence lengths (the tile layout is built on the device); a separate
// instance, since the uniform kernel measured 6 us slower with the ragged branches inlined.
template <int D, int STAGES, int NQB, bool RAGGED>
__global__ void __launch_bounds__(kSThreads, 1) score_kernel(const ScoreParams p,
                                                             const __grid_constant__ CUtensorMap kmap,
                                                             const __grid_constant__ CUtensorMap qmap) {
  constexpr uint32_t KHALF = kSKeys * 128;         // one 64-column half of a K tile
  constexpr uint32_t KTILE = kSKeys * D * 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty_bar = full_bar + STAGES;
  // Accumulator barriers, one pair per epilogue group and not per accumulator: tile i's are
  // those of group i % 4 whatever n_acc.  (Two groups that share an accumulator would each see every
  // second phase of one barrier, and a phase's parity does not tell it from the one two later.)
  uint64_t* tfull_bar = empty_bar + STAGES;        // [kSGroups]
  uint64_t* tempty_bar = tfull_bar + kSGroups;     // [kSGroups]
  uint64_t* qfull_bar = tempty_bar + kSGroups;
  uint64_t* qempty_bar = qfull_bar + 2;
  uint64_t* drain_bar = qempty_bar + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t qbytes = (uint32_t)p.nq_pad * D * 2;
  uint8_t* qbuf = smem + kSQOffset;                            // NQB x qbytes
  uint8_t* kstage = qbuf + NQB * qbytes;                       // STAGES x KTILE (1024-aligned)

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int n_acc = p.n_acc;
  const int n_units = p.total_tiles / p.tiles_per_unit;
  // per-sequence lengths: every CTA lays out the units' middle tiles itself (prefix table
  // after the K stages; the lengths may come from the preceding kernel, so after the
  // dependency wait) and cuts the tile list over the actual tiles
  int* spref = reinterpret_cast<int*>(kstage + STAGES * KTILE);   // [units + 1]
  int total = p.total_tiles, tpc = p.tiles_per_cta;
  if (RAGGED) {
    // with BD_SELECT_WINDOW_READY the lengths were settled before the kernel just before
    // this one too, so the layout (and the streaming) need not wait for it
    if (!p.window_ready) grid_dependency_wait();
    int* wtot = reinterpret_cast<int*>(smem + 1024);
    const int per = (n_units + kSThreads - 1) / kSThreads;
    const int u0 = min(n_units, tid * per), u1 = min(n_units, u0 + per);
    const int tail = p.t_ctx - p.mid_end;            // recent positions
    auto tiles_of = [&](int u) {
      const int t_u = unit_context(p.seq_lens, u, p.h_kv, p.t_ctx, nullptr);
      return (max(0, t_u - tail - p.n_sink) + kSKeys - 1) / kSKeys;
    };
    int sum = 0;
    for (int u = u0; u < u1; ++u) sum += tiles_of(u);
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
      spref[u] = run;
      run += tiles_of(u);
    }
    if (tid == kSThreads - 1) spref[n_units] = run;
    __syncthreads();
    total = spref[n_units];
    tpc = (total + (int)gridDim.x - 1) / (int)gridDim.x;
  }
  const int first = blockIdx.x * tpc;
  const int n = max(0, min(tpc, total - first));
  // Tile g of the list: its unit and its tile within the unit's middle.  Each role walks the
  // list with a unit of its own (unit_first to begin with), moved on past unit ends: a division
  // (or a search of the prefix table) for every tile lengthened the time a K stage is held by
  // the MMA issuer, which bounds the stream.  64 units of 16K in a whole step 175.1 -> 172.8 us,
  // 24 ragged units of up to 36K (a select call) 51.0 -> 46.2 us.
  auto unit_begin = [&](int u) { return RAGGED ? spref[u] : u * p.tiles_per_unit; };
  int unit_first = 0;
  if (RAGGED) {
    int hi = n_units - 1;
    while (unit_first < hi) {
      const int mid = (unit_first + hi + 1) >> 1;
      if (spref[mid] <= first) unit_first = mid;
      else hi = mid - 1;
    }
  } else {
    unit_first = first / p.tiles_per_unit;
  }
  auto locate = [&](int g, int& unit, int& tt) {
    while (g >= unit_begin(unit + 1)) ++unit;
    tt = g - unit_begin(unit);
  };
  auto last_of_unit = [&](int g, int unit) { return g + 1 == unit_begin(unit + 1); };

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int g = 0; g < kSGroups; ++g) {
      mbar_init(&tfull_bar[g], 1);
      mbar_init(&tempty_bar[g], 4);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&qfull_bar[i], 1);
      mbar_init(&qempty_bar[i], 1);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, p.tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    allow_dependent_launch();
    if (lane == 0) {
      tma_prefetch_map(&kmap);
      tma_prefetch_map(&qmap);
    }
    // K tile i into its ring stage (lane 0; false once a wait gave up)
    int k_issued = 0, k_unit = unit_first;
    auto issue_k = [&](int i) -> bool {
      bool ok = true;
      if (lane == 0) {
        int tt;
        locate(first + i, k_unit, tt);
        const int s = i % STAGES;
        if (i >= STAGES) ok = mbar_wait(&empty_bar[s], ((i / STAGES) & 1) ^ 1, p.status, abort_flag);
        if (ok) {
          uint8_t* st = kstage + s * KTILE;
          mbar_arrive_expect_tx(&full_bar[s], KTILE);
          const int key0 = p.n_sink + kSKeys * tt;
#pragma unroll
          for (int h = 0; h < D / 64; ++h) tma_load_3d(st + h * KHALF, &kmap, &full_bar[s], 64 * h, key0, k_unit);
          k_issued = i + 1;
        }
      }
      return __shfl_sync(0xffffffffu, ok, 0);
    };
    // the first stages' K tiles (context rows, which the kernel just before never writes)
    // stream before the grid-dependency wait; the window queries may come from that kernel
    // (bd_advance rewrites them in place), so they load after it, unless the caller says
    // they were written earlier (then queries and tiles interleave from the start)
    const int pre = p.window_ready ? 0 : min(n, STAGES);
    for (int i = 0; i < pre; ++i) issue_k(i);
    if (!p.window_ready) {
      if (n > 0)   // the first unit's queries on their way into L2 meanwhile
        prefetch_lines_l2(p.q_win + (size_t)unit_first * p.nq_rows * D, (size_t)p.nq_rows * D * 2, lane, 32);
      grid_dependency_wait();
    }
    int cur_unit = -1, qcount = 0, unit = unit_first;
    for (int i = 0; i < n; ++i) {
      int tt;
      locate(first + i, unit, tt);
      if (unit != cur_unit) {
        const int qs = qcount % NQB;
        bool ok = true;
        if (lane == 0) {
          // the unit's window-query rows (padded to nq_pad with the next rows, whose scores
          // the epilogue discards) by TMA into the swizzled B-operand tile
          if (qcount >= NQB) ok = mbar_wait(&qempty_bar[qs], ((qcount / NQB) - 1) & 1, p.status, abort_flag);
          if (ok) {
            uint8_t* qb = qbuf + qs * qbytes;
            const uint32_t half_bytes = (uint32_t)p.nq_pad * 128;
            mbar_arrive_expect_tx(&qfull_bar[qs], qbytes);
#pragma unroll
            for (int h = 0; h < D / 64; ++h) tma_load_2d(qb + h * half_bytes, &qmap, &qfull_bar[qs], 64 * h, unit * p.nq_rows);
          }
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) break;
        cur_unit = unit;
        ++qcount;
      }
      if (i >= pre && !issue_k(i)) break;
    }
    if (lane == 0 && *abort_flag) {   // no copy may land in shared memory after the CTA exits
      for (int t = max(0, k_issued - STAGES); t < k_issued; ++t)
        mbar_wait(&full_bar[t % STAGES], (t / STAGES) & 1, p.status, nullptr);
      for (int q = max(0, qcount - NQB); q < qcount; ++q)
        mbar_wait(&qfull_bar[q % NQB], (q / NQB) & 1, p.status, nullptr);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (whole warp, see tc_mma_ss)
    allow_dependent_launch();
    const uint32_t lead = elect_leader();
    const uint32_t idesc = umma_idesc_bf16(kSKeys, p.nq_pad);
    const uint32_t b_half = (uint32_t)p.nq_pad * 128;
    int cur_unit = -1, qcount = 0, unit = unit_first;
    for (int i = 0; i < n; ++i) {
      const int g = first + i;
      int tt;
      locate(g, unit, tt);
      const bool unit_ends = (i == n - 1) || last_of_unit(g, unit);
      if (unit != cur_unit) {
        if (!mbar_wait_warp(&qfull_bar[qcount % NQB], (qcount / NQB) & 1, p.status, abort_flag)) break;
        cur_unit = unit;
        ++qcount;
      }
      const int qs = (qcount - 1) % NQB;
      const int s = i % STAGES;
      const int acc = i % n_acc;
      // the accumulator's tile before this one has been read
      const int prev = i - n_acc;
      if (prev >= 0 && !mbar_wait_warp(&tempty_bar[prev % kSGroups], (prev / kSGroups) & 1, p.status, abort_flag)) break;
      const uint32_t a_lo = desc_k(smem_u32(kstage + s * KTILE));
      const uint32_t b_lo = desc_k(smem_u32(qbuf + qs * qbytes));
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * p.acc_stride);
      if (!mbar_wait_warp(&full_bar[s], (i / STAGES) & 1, p.status, abort_flag)) break;
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks)
        tc_mma_ss(lead, d_tmem, a_lo + ((ks >> 2) * KHALF + (ks & 3) * 32) / 16,
                  b_lo + ((ks >> 2) * b_half + (ks & 3) * 32) / 16, idesc, ks > 0 ? 1u : 0u);
      tc_commit(lead, &empty_bar[s]);
      tc_commit(lead, &tfull_bar[i % kSGroups]);
      if (unit_ends) tc_commit(lead, &qempty_bar[qs]);
    }
    // every MMA this warp issued has completed before TMEM is released
    tc_commit(lead, drain_bar);
    mbar_wait(drain_bar, 0, p.status, nullptr);
  } else {
    // ---------------------------------------------------------------- epilogue (kSGroups groups of 4 warps)
    if (!RAGGED && n > 0 && warp == 2)           // the first unit's window LSE into L2 meanwhile
      prefetch_lines_l2(p.lse_win + (size_t)unit_first * p.nq_rows, (size_t)p.nq_rows * 4, lane, 32);
    grid_dependency_wait();                      // the window LSE is carried from earlier kernels
    allow_dependent_launch();
    const int grp = (warp - 2) >> 2;            // group g: warps 2+4g .. 5+4g; tiles i % 4 == g
    const int quad = warp & 3;                  // TMEM lanes quad*32 .. quad*32+31
    const int ep_tid = (warp - 2 - 4 * grp) * 32 + lane;
    float* lse2_s = reinterpret_cast<float*>(smem + 1024 + grp * 2304);   // [288] -lse * log2(e)
    int* pw_s = reinterpret_cast<int*>(smem + 1024 + grp * 2304 + 1152);  // [288]
    int win0 = p.t_ctx - p.window;              // position of window row 0 (of the current unit)
    int mid_end = p.mid_end;                    // end of the current unit's middle
    int cur_unit = -1, unit = unit_first;
    for (int i = grp; i < n; i += kSGroups) {
      int tt;
      locate(first + i, unit, tt);
      if (unit != cur_unit) {
        if (RAGGED) {
          const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, ep_tid == 0 ? p.status : nullptr);
          if (t_u < p.window && ep_tid == 0) record_error(p.status, BD_ERR_INVALID_ARG);
          win0 = t_u - p.window;
          mid_end = t_u - (p.t_ctx - p.mid_end);
        }
        named_bar(1 + grp, 128);
        for (int c = ep_tid; c < 288; c += 128) {
          const bool real = c < p.nq_rows;
          lse2_s[c] = real ? -__ldg(p.lse_win + (size_t)unit * p.nq_rows + c) * kLog2e : -INFINITY;
          pw_s[c] = real ? win0 + c % p.window : -1;
        }
        named_bar(1 + grp, 128);
        cur_unit = unit;
      }
      const int acc = i % n_acc;
      if (!mbar_wait(&tfull_bar[grp], (i / kSGroups) & 1, p.status, abort_flag)) break;
      tc_fence_after();
      const int key_tile0 = p.n_sink + kSKeys * tt;
      const int key = key_tile0 + quad * 32 + lane;
      const bool causal = key_tile0 + kSKeys - 1 > win0;   // some key may follow a window row
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * p.acc_stride);
      float sum0 = 0.f, sum1 = 0.f, sum2 = 0.f, sum3 = 0.f;
      for (int c0 = 0; c0 < p.nq_pad; c0 += 64) {
        float v[64];
        tc_ld_32cols(taddr + c0, *reinterpret_cast<float(*)[32]>(&v[0]));
        tc_ld_32cols(taddr + c0 + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
        tc_wait_ld();
        const int ncol = min(64, p.nq_pad - c0);
        if (ncol == 64 && !causal) {
          // packed pairs: one f32x2 FMA and one f32x2 add per two scores (the epilogue's
          // instruction issue, not the exponentials, limits this loop)
          const float2 cc = make_float2(p.scale_log2, p.scale_log2);
          float2 a0 = make_float2(0.f, 0.f), a1 = a0, a2 = a0, a3 = a0;
#pragma unroll
          for (int j = 0; j < 64; j += 8) {
            const float4 la = *reinterpret_cast<const float4*>(lse2_s + c0 + j);
            const float4 lb = *reinterpret_cast<const float4*>(lse2_s + c0 + j + 4);
            const float2 x0 = ffma2(make_float2(v[j], v[j + 1]), cc, make_float2(la.x, la.y));
            const float2 x1 = ffma2(make_float2(v[j + 2], v[j + 3]), cc, make_float2(la.z, la.w));
            const float2 x2 = ffma2(make_float2(v[j + 4], v[j + 5]), cc, make_float2(lb.x, lb.y));
            const float2 x3 = ffma2(make_float2(v[j + 6], v[j + 7]), cc, make_float2(lb.z, lb.w));
            a0 = fadd2(a0, make_float2(fast_exp2(x0.x), fast_exp2(x0.y)));
            a1 = fadd2(a1, make_float2(fast_exp2(x1.x), fast_exp2(x1.y)));
            a2 = fadd2(a2, make_float2(fast_exp2(x2.x), fast_exp2(x2.y)));
            a3 = fadd2(a3, make_float2(fast_exp2(x3.x), fast_exp2(x3.y)));
          }
          sum0 += a0.x + a0.y;
          sum1 += a1.x + a1.y;
          sum2 += a2.x + a2.y;
          sum3 += a3.x + a3.y;
        } else {
#pragma unroll
          for (int j = 0; j < 64; ++j) {
            if (j < ncol) {
              const float x = key <= pw_s[c0 + j] ? fmaf(v[j], p.scale_log2, lse2_s[c0 + j]) : -INFINITY;
              sum0 += fast_exp2(x);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&tempty_bar[grp]);
      // (a NaN, from one in a key, a query or a normaliser, counts as 0: ranked by its bits it would be above
      // every threshold while the histogram has it in the lowest bin, and more items than the budget holds
      // would be written)
      if (key < mid_end)
        p.score[(size_t)unit * p.n_mid_pad + (key - p.n_sink)] = fmaxf((sum0 + sum1) + (sum2 + sum3), 0.f);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, p.tmem_cols);
}

// ============================================================================ window LSE
//
// Self mode's normalisers, and bd_verify_attn without an output: lse_r = log sum_{k <= p_w} exp(q_r . k_k / sqrt(d)) for the G*W
// window rows r = h*W + w of every unit (p_w = t_ctx - W + w).  The contraction of
// score_kernel with its operands swapped: the unit's window rows are the A operand (M =
// 128 rows = the TMEM lanes) and a 128-key K tile the B operand (N = 128 columns), so a
// row's online log-sum-exp stays inside the two threads that own it (one per 64-column
// half of the TMEM row), with no reduction across lanes.  Persistent CTAs (one per SM)
// take contiguous ranges of the (unit, 128-key tile) list: warp 0 streams K tiles (TMA,
// 4-stage ring) and the unit's rows (two buffers), warp 1 issues the MMAs into four TMEM
// accumulators, warps 2-9 reduce (two warps per TMEM lane quarter).  A unit split over
// several CTAs merges the segments' (max, sum) pairs in the CTA that finishes it last.
// HBM-bound: 268 MB of K (64 units of 16K, 128 rows each) in 46.5 us, 5.8 TB/s; the same rows as
// an mma.sync verify block without V took 124 us, bound by the tensor pipe.  With up to 64 rows the
// operand holds them two or four times (COPIES): 128 units of 16K, 32 rows, d 64 68.3 us with one copy
// (one lane quarter computes all the exponentials that count), 48.6 with four; d 128 82.1 / 78.9.
struct LseParams {
  const __nv_bfloat16* q_win;   // [units * nq_rows][D] (read by TMA; prefetched through this pointer)
  float* lse;          // [units * nq_rows] natural log
  float2* part;        // [units][max_seg][128]: a segment's (running max in log2 units, sum)
  int* counters;       // [units] arrival counters (left zero)
  int* status;
  int nq_rows, window, t_ctx, tiles_per_unit, total_tiles, tiles_per_cta, max_seg;
  int settled;         // rows [0, settled) of every unit are older than the preceding kernel
  int window_ready;    // BD_SELECT_WINDOW_READY: the rows may load before the dependency wait
  float scale_log2;
  const int32_t* seq_lens;   // per-sequence context lengths [batch] (RAGGED instance) or null
  int len_offset;            // added to every length (a verify block ends n_q past its context)
  int h_kv, units;
};
// Segments of one unit with per-sequence lengths (bounds the partials): 33 while the units are not many
// times the SMs, since all but a few sequences may be short.  (One sequence of 64K, 8 units of 24 or 32 rows:
// 53.5 us with 8 segments.)
constexpr int kLMinSeg = 8, kLMaxSeg = 33;
constexpr int kLThreads = 320;   // producer, MMA, eight epilogue warps (two per TMEM lane quarter)
constexpr int kLAcc = 4;         // TMEM accumulators of 128 columns
constexpr int kLStages = 4;

// RAGGED: per-sequence lengths; every CTA lays out the units' tiles itself (a prefix table in
// shared memory, as score_kernel's ragged instance does) and the range per CTA is at least
// tiles_per_cta, which keeps a unit within max_seg segments.
constexpr float kLn2Rest = -1.9046542e-9f;   // ln 2 less kLn2
// log(2^m l) for a whole number m: the logarithm of l's fraction alone is rounded before the last sum (that
// of l itself, 5 or so, by half as much as the result).
__device__ __forceinline__ float row_lse(float m, float l) {
  if (!(l > 0.f)) return -INFINITY;
  int e;
  const float f = frexpf(l, &e);
  const float x = m + (float)e;
  return fmaf(x, kLn2, fmaf(x, kLn2Rest, logf(f)));
}

// COPIES: how often the unit's rows (at most 128 / COPIES) lie in the A operand, each copy taking its share
// of a tile's columns: a quarter of the lanes holding all the rows would have all the exponentials.
template <int D, bool RAGGED, int COPIES>
__global__ void __launch_bounds__(kLThreads, 1) window_lse_kernel(const LseParams p,
                                                                  const __grid_constant__ CUtensorMap kmap,
                                                                  const __grid_constant__ CUtensorMap qmap) {
  constexpr int STAGES = kLStages;
  constexpr uint32_t KHALF = kSKeys * 128;   // one 64-column half of a K tile
  constexpr uint32_t KTILE = kSKeys * D * 2;
  constexpr uint32_t QHALF = 128 * 128;      // one 64-column half of the 128 window rows
  constexpr uint32_t QTILE = 128 * D * 2;
  constexpr int ROWS = 128 / COPIES;         // rows of a copy
  constexpr int COLS = 64 / COPIES;          // columns of a tile per epilogue thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem);
  uint64_t* empty_bar = full_bar + STAGES;
  uint64_t* tfull_bar = empty_bar + STAGES;    // [kLAcc]
  uint64_t* tempty_bar = tfull_bar + kLAcc;    // [kLAcc]
  uint64_t* qfull_bar = tempty_bar + kLAcc;    // [2]
  uint64_t* qempty_bar = qfull_bar + 2;        // [2]
  uint64_t* drain_bar = qempty_bar + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* last_flag = const_cast<int*>(abort_flag) + 1;
  uint8_t* qbuf = smem + 1024;                 // 2 x QTILE
  uint8_t* kstage = qbuf + 2 * QTILE;          // STAGES x KTILE
  float2* ml_s = reinterpret_cast<float2*>(kstage + STAGES * KTILE);   // [2][128] the column halves' (m, l)
  int* spref = reinterpret_cast<int*>(ml_s + 256);                      // [units + 1] (RAGGED)

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  const int tpu = p.tiles_per_unit;
  int total = p.total_tiles, tpc = p.tiles_per_cta;
  if (RAGGED) {
    // the lengths may come from the kernel just before (bd_advance moves them), unless the
    // caller says otherwise
    if (!p.window_ready) grid_dependency_wait();
    int* wtot = reinterpret_cast<int*>(smem + 512);
    const int per = (p.units + kLThreads - 1) / kLThreads;
    const int u0 = min(p.units, tid * per), u1 = min(p.units, u0 + per);
    auto tiles_of = [&](int u) {
      return (unit_context(p.seq_lens, u, p.h_kv, p.t_ctx - p.len_offset, nullptr) + p.len_offset + kSKeys - 1) / kSKeys;
    };
    int sum = 0;
    for (int u = u0; u < u1; ++u) sum += tiles_of(u);
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
      spref[u] = run;
      run += tiles_of(u);
    }
    if (tid == kLThreads - 1) spref[p.units] = run;
    __syncthreads();
    total = spref[p.units];
    tpc = max((total + (int)gridDim.x - 1) / (int)gridDim.x, p.tiles_per_cta);
  }
  const int first = blockIdx.x * tpc;
  const int n = max(0, min(tpc, total - first));
  auto unit_begin = [&](int u) { return RAGGED ? spref[u] : u * tpu; };
  auto unit_end = [&](int u) { return unit_begin(u + 1); };
  // the unit of the range's first tile; each role walks on from it (as in score_kernel)
  int unit_first = 0;
  if (RAGGED) {
    int hi = p.units - 1;
    while (unit_first < hi) {
      const int mid = (unit_first + hi + 1) >> 1;
      if (spref[mid] <= first) unit_first = mid;
      else hi = mid - 1;
    }
  } else {
    unit_first = first / tpu;
  }
  auto walk = [&](int g, int& unit) {
    while (g >= unit_end(unit)) ++unit;
  };

  if (tid == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < kLAcc; ++a) {
      mbar_init(&tfull_bar[a], 1);
      mbar_init(&tempty_bar[a], 8);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&qfull_bar[i], 1);
      mbar_init(&qempty_bar[i], 1);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kLAcc * 128);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    allow_dependent_launch();
    if (lane == 0) {
      tma_prefetch_map(&kmap);
      tma_prefetch_map(&qmap);
    }
    int k_issued = 0, k_unit = unit_first;
    auto issue_k = [&](int i) -> bool {
      bool ok = true;
      if (lane == 0) {
        walk(first + i, k_unit);
        const int tt = first + i - unit_begin(k_unit);
        const int s = i % STAGES;
        if (i >= STAGES) ok = mbar_wait(&empty_bar[s], ((i / STAGES) & 1) ^ 1, p.status, abort_flag);
        if (ok) {
          uint8_t* st = kstage + s * KTILE;
          mbar_arrive_expect_tx(&full_bar[s], KTILE);
#pragma unroll
          for (int h = 0; h < D / 64; ++h) tma_load_3d(st + h * KHALF, &kmap, &full_bar[s], 64 * h, kSKeys * tt, k_unit);
          k_issued = i + 1;
        }
      }
      return __shfl_sync(0xffffffffu, ok, 0);
    };
    // K tiles of settled rows stream before the grid-dependency wait (with per-sequence lengths
    // the wait came first); the window rows after it (before it as well when the caller says
    // they were written earlier)
    int pre = 0;
    if (!p.window_ready) {
      int u = unit_first;
      auto old_rows = [&](int i) {
        walk(first + i, u);
        return kSKeys * (first + i - unit_begin(u) + 1) <= p.settled;
      };
      for (; pre < min(n, STAGES) && (RAGGED || old_rows(pre)); ++pre) issue_k(pre);
      if (n > 0)   // the first unit's rows on their way into L2 meanwhile
        prefetch_lines_l2(p.q_win + (size_t)unit_first * p.nq_rows * D, (size_t)p.nq_rows * D * 2, lane, 32);
      grid_dependency_wait();
    }
    int cur_unit = -1, qcount = 0, unit = unit_first;
    for (int i = 0; i < n; ++i) {
      walk(first + i, unit);
      if (unit != cur_unit) {
        const int qs = qcount & 1;
        bool ok = true;
        if (lane == 0) {
          // rows unit*nq_rows .. + ROWS - 1 (past nq_rows: the next unit's rows or zero fill, whose
          // results are discarded)
          if (qcount >= 2) ok = mbar_wait(&qempty_bar[qs], ((qcount >> 1) - 1) & 1, p.status, abort_flag);
          if (ok) {
            uint8_t* qb = qbuf + qs * QTILE;
            mbar_arrive_expect_tx(&qfull_bar[qs], QTILE);
#pragma unroll
            for (int h = 0; h < D / 64; ++h)
#pragma unroll
              for (int c = 0; c < COPIES; ++c)
                tma_load_2d(qb + h * QHALF + c * ROWS * 128, &qmap, &qfull_bar[qs], 64 * h, unit * p.nq_rows);
          }
        }
        if (!__shfl_sync(0xffffffffu, ok, 0)) break;
        cur_unit = unit;
        ++qcount;
      }
      if (i >= pre && !issue_k(i)) break;
    }
    if (lane == 0 && *abort_flag) {   // no copy may land in shared memory after the CTA exits
      for (int t = max(0, k_issued - STAGES); t < k_issued; ++t)
        mbar_wait(&full_bar[t % STAGES], (t / STAGES) & 1, p.status, nullptr);
      for (int q = max(0, qcount - 2); q < qcount; ++q) mbar_wait(&qfull_bar[q & 1], (q >> 1) & 1, p.status, nullptr);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (whole warp, see tc_mma_ss)
    allow_dependent_launch();
    const uint32_t lead = elect_leader();
    constexpr uint32_t idesc = umma_idesc_bf16(128, kSKeys);
    int cur_unit = -1, qcount = 0, unit = unit_first;
    for (int i = 0; i < n; ++i) {
      const int g = first + i;
      walk(g, unit);
      const bool unit_ends = (i == n - 1) || g + 1 == unit_end(unit);
      if (unit != cur_unit) {
        if (!mbar_wait_warp(&qfull_bar[qcount & 1], (qcount >> 1) & 1, p.status, abort_flag)) break;
        cur_unit = unit;
        ++qcount;
      }
      const int qs = (qcount - 1) & 1;
      const int s = i % STAGES;
      const int acc = i % kLAcc;
      if (i >= kLAcc && !mbar_wait_warp(&tempty_bar[acc], ((i / kLAcc) & 1) ^ 1, p.status, abort_flag)) break;
      const uint32_t a_lo = desc_k(smem_u32(qbuf + qs * QTILE));
      const uint32_t b_lo = desc_k(smem_u32(kstage + s * KTILE));
      const uint32_t d_tmem = tmem_base + (uint32_t)(acc * 128);
      if (!mbar_wait_warp(&full_bar[s], (i / STAGES) & 1, p.status, abort_flag)) break;
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks)
        tc_mma_ss(lead, d_tmem, a_lo + ((ks >> 2) * QHALF + (ks & 3) * 32) / 16,
                  b_lo + ((ks >> 2) * KHALF + (ks & 3) * 32) / 16, idesc, ks > 0 ? 1u : 0u);
      tc_commit(lead, &empty_bar[s]);
      tc_commit(lead, &tfull_bar[acc]);
      if (unit_ends) tc_commit(lead, &qempty_bar[qs]);
    }
    tc_commit(lead, drain_bar);
    mbar_wait(drain_bar, 0, p.status, nullptr);
  } else {
    // ---------------------------------------------------------------- epilogue: COLS columns of a row per thread
    grid_dependency_wait();
    allow_dependent_launch();
    const int quad = warp & 3;                  // TMEM lanes quad*32 .. quad*32+31
    const int half = (warp - 2) >> 2;           // warps 2-5: columns 0-63, warps 6-9: 64-127
    const int copy = quad * 32 / ROWS, row = quad * 32 + lane - copy * ROWS;
    const bool first_copy = half == 0 && copy == 0;       // merges and writes its row
    int pw = p.t_ctx - p.window + row % p.window;         // last key the row sees
    int first_masked = p.t_ctx - p.window;                // keys past it are hidden from some row
    int cur_unit = -1, unit = unit_first;
    float m = -INFINITY, l = 0.f;                          // log2 units
    // after a wait gives up, a warp keeps walking its tiles without touching TMEM, so that
    // all eight warps still meet at every unit-end barrier
    bool alive = true;
    for (int i = 0; i < n; ++i) {
      const int g = first + i;
      walk(g, unit);
      const int tt = g - unit_begin(unit);
      if (RAGGED && unit != cur_unit) {
        const int t_u =
            unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx - p.len_offset, tid == 64 ? p.status : nullptr) + p.len_offset;
        if (t_u < p.window && tid == 64) record_error(p.status, BD_ERR_INVALID_ARG);
        pw = t_u - p.window + row % p.window;
        first_masked = t_u - p.window;
        cur_unit = unit;
      }
      const int acc = i % kLAcc;
      alive = __all_sync(0xffffffffu, alive && mbar_wait(&tfull_bar[acc], (i / kLAcc) & 1, p.status, abort_flag));
      if (alive) {
        tc_fence_after();
        const int key0 = kSKeys * tt;
        const bool masked = key0 + kSKeys - 1 > first_masked;
        const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 128);
        {
          const int c0 = 64 * half + COLS * copy;
          float v[COLS];
          if constexpr (COLS == 16) {
            tc_ld_16cols(taddr + c0, v);
          } else {
#pragma unroll
            for (int j = 0; j < COLS; j += 32) tc_ld_32cols(taddr + c0 + j, *reinterpret_cast<float(*)[32]>(&v[j]));
          }
          tc_wait_ld();
          if (masked) {
#pragma unroll
            for (int j = 0; j < COLS; ++j) v[j] = key0 + c0 + j <= pw ? v[j] : -INFINITY;
          }
          float mx0 = fmaxf(v[0], v[1]), mx1 = fmaxf(v[2], v[3]);
#pragma unroll
          for (int j = 4; j < COLS; j += 4) {
            mx0 = fmaxf(mx0, fmaxf(v[j], v[j + 1]));
            mx1 = fmaxf(mx1, fmaxf(v[j + 2], v[j + 3]));
          }
          const float mxs = fmaxf(mx0, mx1) * p.scale_log2;
          if (mxs > m) {
            // rounded up to a whole number, so that sums under different maxima meet by exact powers of two
            // (by additions: ceilf shares a unit with the exponentials, 39.4 us for 64 units of 16K, d 64, against 38.9)
            const float up = __fadd_ru(mxs, 12582912.f) - 12582912.f;
            l *= fast_exp2(m - up);                  // m = -inf: l is still 0
            m = up;
          }
          const float2 cc = make_float2(p.scale_log2, p.scale_log2);
          const float2 nm = make_float2(m == -INFINITY ? 0.f : -m, m == -INFINITY ? 0.f : -m);
          float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
          for (int j = 0; j < COLS; j += 4) {
            const float2 x0 = ffma2(make_float2(v[j], v[j + 1]), cc, nm);
            const float2 x1 = ffma2(make_float2(v[j + 2], v[j + 3]), cc, nm);
            a0 = fadd2(a0, make_float2(fast_exp2(x0.x), fast_exp2(x0.y)));
            a1 = fadd2(a1, make_float2(fast_exp2(x1.x), fast_exp2(x1.y)));
          }
          l += (a0.x + a0.y) + (a1.x + a1.y);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty_bar[acc]);
      }
      if (i != n - 1 && g + 1 != unit_end(unit)) continue;
      // ------------------------------------------------------------ end of this CTA's part of the unit
      // a row's column shares meet first
      ml_s[(half * COPIES + copy) * ROWS + row] = alive ? make_float2(m, l) : make_float2(-INFINITY, 0.f);
      named_bar(1, 256);
      const int c_first = unit_begin(unit) / tpc, c_last = (unit_end(unit) - 1) / tpc;
      const int n_seg = c_last - c_first + 1;
      const size_t row0 = (size_t)unit * p.nq_rows;
      float2* seg = p.part + (size_t)unit * p.max_seg * 128;
      if (first_copy) {
#pragma unroll
        for (int h = 1; h < 2 * COPIES; ++h) {
          const float2 o = ml_s[h * ROWS + row];
          const float M2 = fmaxf(m, o.x);
          l = (m == -INFINITY ? 0.f : l * fast_exp2(m - M2)) + (o.x == -INFINITY ? 0.f : o.y * fast_exp2(o.x - M2));
          m = M2;
        }
        if (n_seg == 1) {
          if (alive && row < p.nq_rows) p.lse[row0 + row] = row_lse(m, l);
        } else if (alive) {
          seg[(size_t)((int)blockIdx.x - c_first) * 128 + row] = make_float2(m, l);
        }
      }
      if (n_seg > 1) {
        __threadfence();
        named_bar(1, 256);
        if (first_copy && row == 0) *last_flag = alive && atomicAdd(&p.counters[unit], 1) == n_seg - 1;
        named_bar(1, 256);
        if (first_copy && *last_flag) {
          __threadfence();
          float M = -INFINITY;
          for (int k = 0; k < n_seg; ++k) M = fmaxf(M, __ldcg(&seg[(size_t)k * 128 + row].x));
          float L = 0.f;
          for (int k = 0; k < n_seg; ++k) {
            const float2 ml = __ldcg(&seg[(size_t)k * 128 + row]);
            L += ml.x == -INFINITY ? 0.f : ml.y * fast_exp2(ml.x - M);
          }
          if (row < p.nq_rows) p.lse[row0 + row] = row_lse(M, L);
          if (row == 0) p.counters[unit] = 0;
        }
      }
      named_bar(1, 256);                          // ml_s and last_flag are free for the next unit
      m = -INFINITY;
      l = 0.f;
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, kLAcc * 128);
}

// ============================================================================ top-B select

// Token-level selection with the scores staged in shared memory: the register kernels'
// method for middles of up to 32K where the batch leaves no SMs for a cluster per unit.
// Needs 0 < k < n <= kLeanMaxItems; the selection mask of each item is kept as warp ballots
// in registers.
constexpr int kLeanMaxItems = 32 * kTopkThreads;   // 32 rows of 32 items per warp
constexpr int kLeanRows = kLeanMaxItems / kTopkThreads;

__global__ void __launch_bounds__(kTopkThreads, 1) topk_token_kernel(const TopkParams p) {
  extern __shared__ uint32_t vals[];                // n scores (fp32 bits)
  __shared__ uint32_t bins[kBins];
  __shared__ uint64_t cand[kBinCandMax];
  __shared__ uint32_t wsum[32];
  __shared__ float wmin[32], wmax[32];
  __shared__ uint32_t s_total, s_bin, s_above, s_nc, s_taukey, s_eq_take, s_eq_all, s_prefix, s_krem;
  __shared__ float s_vmin, s_vmax;
  grid_dependency_wait();
  allow_dependent_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = blockIdx.x;
  const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 ? p.status : nullptr);
  int32_t* out = p.idx_out + (size_t)unit * p.budget;
  if (topk_keep_all(p, unit, t_u, out, tid, kTopkThreads)) return;
  const int lo = p.n_sink, hi = t_u - p.n_recent, n = hi - lo;
  const int k = p.budget - p.n_sink - p.n_recent;
  const float* sc = p.score + (size_t)unit * p.n_mid_pad;

  // ---- stage the scores, min and max
  float lmin = INFINITY, lmax = -INFINITY;
  const int n4 = n >> 2;
  const float4* sc4 = reinterpret_cast<const float4*>(sc);
  for (int i = tid; i < n4; i += kTopkThreads) {
    const float4 v = __ldcg(sc4 + i);
    reinterpret_cast<uint4*>(vals)[i] = make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z),
                                                   __float_as_uint(v.w));
    lmin = fminf(fminf(lmin, fminf(v.x, v.y)), fminf(v.z, v.w));
    lmax = fmaxf(fmaxf(lmax, fmaxf(v.x, v.y)), fmaxf(v.z, v.w));
  }
  for (int i = 4 * n4 + tid; i < n; i += kTopkThreads) {
    const float v = __ldcg(sc + i);
    vals[i] = __float_as_uint(v);
    lmin = fminf(lmin, v);
    lmax = fmaxf(lmax, v);
  }
  for (int i = tid; i < kBins; i += kTopkThreads) bins[i] = 0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, off));
    lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
  }
  if (lane == 0) {
    wmin[warp] = lmin;
    wmax[warp] = lmax;
  }
  if (tid == 0) {
    s_nc = 0;
    s_eq_take = 0;
    s_eq_all = 0;
  }
  __syncthreads();
  if (warp == 0) {
    float a = wmin[lane], b = wmax[lane];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      a = fminf(a, __shfl_xor_sync(0xffffffffu, a, off));
      b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, off));
    }
    if (lane == 0) {
      s_vmin = a;
      s_vmax = b;
    }
  }
  __syncthreads();
  const float vmin = s_vmin, vmax = s_vmax;

  // ---- tau (bits of the k-th largest score) and krem (how many scores equal to tau to keep)
  uint32_t tau = 0, krem = (uint32_t)k;
  bool simple = false, found = false;
  if (vmax > vmin) {
    const float scale = (float)(kBins - 1) / (vmax - vmin);
    auto bin_of = [&](uint32_t u) -> int { return min(kBins - 1, (int)((__uint_as_float(u) - vmin) * scale)); };
    for (int i = tid; i < n; i += kTopkThreads) atomicAdd(&bins[bin_of(vals[i])], 1u);
    __syncthreads();
    constexpr int BPT = kBins / kTopkThreads;
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < BPT; ++j) mine += bins[tid * BPT + j];
    uint32_t incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += z;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = wsum[lane];
      uint32_t c = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
        if (lane >= off) c += z;
      }
      wsum[lane] = c - w;
      if (lane == 31) s_total = c;
    }
    __syncthreads();
    uint32_t above = s_total - (wsum[warp] + incl);
#pragma unroll
    for (int j = BPT - 1; j >= 0; --j) {
      const uint32_t h = bins[tid * BPT + j];
      if (above < (uint32_t)k && (uint32_t)k <= above + h) {
        s_bin = (uint32_t)(tid * BPT + j);
        s_above = above;
      }
      above += h;
    }
    __syncthreads();
    const int bstar = (int)s_bin;
    const uint32_t nc = bins[bstar];
    if (nc <= (uint32_t)kBinCandMax) {
      for (int i = tid; i < n; i += kTopkThreads) {
        const uint32_t u = vals[i];
        if (bin_of(u) == bstar) cand[atomicAdd(&s_nc, 1u)] = (static_cast<uint64_t>(u) << 32) | (0xFFFFFFFFu - (uint32_t)i);
      }
      __syncthreads();
      const uint32_t m = (uint32_t)k - s_above;
      uint64_t key = 0;
      uint32_t rank = 0xFFFFFFFFu;
      if (tid < (int)nc) {
        key = cand[tid];
        rank = 0;
        for (int j = 0; j < (int)nc; ++j) rank += cand[j] > key;
        if (rank == m - 1) s_taukey = static_cast<uint32_t>(key >> 32);
      }
      for (int i = tid + kTopkThreads; i < (int)nc; i += kTopkThreads) {   // nc > 1024: rare
        const uint64_t kk = cand[i];
        uint32_t r = 0;
        for (int j = 0; j < (int)nc; ++j) r += cand[j] > kk;
        if (r == m - 1) s_taukey = static_cast<uint32_t>(kk >> 32);
      }
      __syncthreads();
      tau = s_taukey;
      for (int i = tid; i < (int)nc; i += kTopkThreads) {
        const uint64_t kk = cand[i];
        if (static_cast<uint32_t>(kk >> 32) != tau) continue;
        uint32_t r = (i == tid) ? rank : 0;
        if (i != tid)
          for (int j = 0; j < (int)nc; ++j) r += cand[j] > kk;
        atomicAdd(&s_eq_all, 1u);
        if (r < m) atomicAdd(&s_eq_take, 1u);
      }
      __syncthreads();
      krem = s_eq_take;
      simple = (s_eq_take == s_eq_all);
      found = true;
    }
  }
  if (!found) {
    // crowded boundary (many equal or near-equal scores): exact 4-pass radix select
    uint32_t prefix = 0, mask = 0;
    krem = (uint32_t)k;
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = tid; i < 256; i += kTopkThreads) bins[i] = 0;
      __syncthreads();
      for (int i = tid; i < n; i += kTopkThreads) {
        const uint32_t u = vals[i];
        if ((u & mask) == prefix) atomicAdd(&bins[(u >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (warp == 0) {
        uint32_t local = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) local += bins[8 * lane + j];
        uint32_t suffix = local;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t y = __shfl_down_sync(0xffffffffu, suffix, off);
          if (lane + off < 32) suffix += y;
        }
        uint32_t abv = suffix - local;
        if (abv < krem && krem <= suffix) {
          for (int j = 7; j >= 0; --j) {
            const uint32_t h = bins[8 * lane + j];
            if (abv + h >= krem) {
              s_prefix = prefix | ((uint32_t)(8 * lane + j) << shift);
              s_krem = krem - abv;
              break;
            }
            abv += h;
          }
        }
      }
      __syncthreads();
      prefix = s_prefix;
      krem = s_krem;
      mask |= 0xFFu << shift;
    }
    tau = prefix;
    simple = false;
  }

  // ---- ascending compaction: warp w owns items [w*ipw, (w+1)*ipw), rows of 32
  const int rows = (n + kTopkThreads - 1) / kTopkThreads;     // <= kLeanRows
  const int w0 = warp * rows * 32;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t eq_base = 0;
  if (!simple) {
    uint32_t eqc = 0;
#pragma unroll
    for (int r = 0; r < kLeanRows; ++r) {
      if (r < rows) {
        const int i = w0 + 32 * r + lane;
        eqc += __popc(__ballot_sync(0xffffffffu, i < n && vals[i] == tau));
      }
    }
    if (lane == 0) wsum[warp] = eqc;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = wsum[lane];
      uint32_t c = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
        if (lane >= off) c += z;
      }
      wsum[lane] = c - w;
    }
    __syncthreads();
    eq_base = wsum[warp];
    __syncthreads();
  }
  uint32_t masks[kLeanRows];
  uint32_t cnt = 0, eq_run = eq_base;
#pragma unroll
  for (int r = 0; r < kLeanRows; ++r) {
    masks[r] = 0;
    if (r < rows) {
      const int i = w0 + 32 * r + lane;
      const uint32_t u = i < n ? vals[i] : 0u;
      bool sel = i < n && u > tau;
      const bool eq = i < n && u == tau;
      if (simple) {
        sel |= eq;
      } else {
        const uint32_t be = __ballot_sync(0xffffffffu, eq);
        if (eq) sel = eq_run + __popc(be & lt) < krem;
        eq_run += __popc(be);
      }
      masks[r] = __ballot_sync(0xffffffffu, sel);
      cnt += __popc(masks[r]);
    }
  }
  if (lane == 0) wsum[warp] = cnt;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = wsum[lane];
    uint32_t c = w;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
      if (lane >= off) c += z;
    }
    wsum[lane] = c - w;
    if (lane == 31) s_total = c;
  }
  __syncthreads();
  uint32_t base = (uint32_t)lo + wsum[warp];
#pragma unroll
  for (int r = 0; r < kLeanRows; ++r) {
    if (r < rows) {
      const uint32_t mk = masks[r];
      if ((mk >> lane) & 1u) out[base + __popc(mk & lt)] = lo + w0 + 32 * r + lane;
      base += __popc(mk);
    }
  }
  const int n_chosen = (int)s_total;
  const int count = lo + n_chosen + p.n_recent;
  for (int i = tid; i < lo; i += kTopkThreads) out[i] = i;
  for (int i = tid; i < p.n_recent; i += kTopkThreads) out[lo + n_chosen + i] = hi + i;
  for (int i = count + tid; i < p.budget; i += kTopkThreads) out[i] = -1;
  if (tid == 0) p.count_out[unit] = count;
}

// Shared storage of the register-resident top-B kernels.
struct TopkRowsSmem {
  uint32_t bins[kBins];
  uint64_t cand[kBinCandMax];
  uint32_t wsum[32], wpos[32];
  float wmin[32], wmax[32];
  uint32_t s_total, s_bin, s_above, s_nc, s_taukey, s_eq_take, s_eq_all, s_prefix, s_krem;
};

// The k-th largest of the block's items: tau (its fp32 bits), krem (how many items equal to
// tau are kept, in item order) and whether that is all of them.
struct RowsThreshold {
  uint32_t tau, krem;
  bool simple;
};

// Items in registers, ROWS per thread: warp w owns items [w*ROWS*32, (w+1)*ROWS*32), row r of
// it at w*ROWS*32 + 32r + lane; values are fp32 bits of non-negative scores (the order of the
// bits), +0 in slots past the item count (no item is below it and ties go to the lower item,
// so the padding never displaces an item).  A linear histogram between the smallest and the
// largest value (lmin, lmax: this thread's) finds the bin of the k-th value and its items are
// ranked exactly; a crowded bin takes an exact 4-pass radix select on the bits.  0 < k < n.
template <int ROWS>
__device__ __forceinline__ RowsThreshold rows_threshold(TopkRowsSmem& S, const uint32_t (&u)[ROWS], float lmin,
                                                        float lmax, int k) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int w0 = warp * ROWS * 32;
  for (int i = tid; i < kBins; i += kTopkThreads) S.bins[i] = 0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, off));
    lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
  }
  if (lane == 0) {
    S.wmin[warp] = lmin;
    S.wmax[warp] = lmax;
  }
  if (tid == 0) {
    S.s_nc = 0;
    S.s_eq_take = 0;
    S.s_eq_all = 0;
  }
  __syncthreads();
  float vmin = S.wmin[lane], vmax = S.wmax[lane];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    vmin = fminf(vmin, __shfl_xor_sync(0xffffffffu, vmin, off));
    vmax = fmaxf(vmax, __shfl_xor_sync(0xffffffffu, vmax, off));
  }

  // ---- tau (bits of the k-th largest score) and krem (how many scores equal to tau to keep)
  uint32_t tau = 0, krem = (uint32_t)k;
  bool simple = false, found = false;
  if (vmax > vmin) {
    const float scale = (float)(kBins - 1) / (vmax - vmin);
    auto bin_of = [&](uint32_t x) -> int { return min(kBins - 1, (int)((__uint_as_float(x) - vmin) * scale)); };
#pragma unroll
    for (int r = 0; r < ROWS; ++r) atomicAdd(&S.bins[bin_of(u[r])], 1u);
    __syncthreads();
    constexpr int BPT = kBins / kTopkThreads;
    uint32_t hb[BPT];
    const uint4 hv = reinterpret_cast<const uint4*>(S.bins)[tid];
    hb[0] = hv.x;
    hb[1] = hv.y;
    hb[2] = hv.z;
    hb[3] = hv.w;
    uint32_t incl = hb[0] + hb[1] + hb[2] + hb[3];
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += z;
    }
    if (lane == 31) S.wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = S.wsum[lane];
      uint32_t c = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
        if (lane >= off) c += z;
      }
      S.wsum[lane] = c - w;
      if (lane == 31) S.s_total = c;
    }
    __syncthreads();
    uint32_t above = S.s_total - (S.wsum[warp] + incl);
#pragma unroll
    for (int j = BPT - 1; j >= 0; --j) {
      if (above < (uint32_t)k && (uint32_t)k <= above + hb[j]) {
        S.s_bin = (uint32_t)(tid * BPT + j);
        S.s_above = above;
        S.s_prefix = hb[j];
      }
      above += hb[j];
    }
    __syncthreads();
    const int bstar = (int)S.s_bin;
    const uint32_t nc = S.s_prefix;
    if (nc <= (uint32_t)kBinCandMax) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int i = w0 + 32 * r + lane;
        if (bin_of(u[r]) == bstar)
          S.cand[atomicAdd(&S.s_nc, 1u)] = (static_cast<uint64_t>(u[r]) << 32) | (0xFFFFFFFFu - (uint32_t)i);
      }
      __syncthreads();
      const uint32_t m = (uint32_t)k - S.s_above;
      for (int i = tid; i < (int)nc; i += kTopkThreads) {
        const uint64_t kk = S.cand[i];
        uint32_t rk = 0;
        for (int j = 0; j < (int)nc; ++j) rk += S.cand[j] > kk;
        if (rk == m - 1) S.s_taukey = static_cast<uint32_t>(kk >> 32);
      }
      __syncthreads();
      tau = S.s_taukey;
      for (int i = tid; i < (int)nc; i += kTopkThreads) {
        const uint64_t kk = S.cand[i];
        if (static_cast<uint32_t>(kk >> 32) != tau) continue;
        uint32_t rk = 0;
        for (int j = 0; j < (int)nc; ++j) rk += S.cand[j] > kk;
        atomicAdd(&S.s_eq_all, 1u);
        if (rk < m) atomicAdd(&S.s_eq_take, 1u);
      }
      __syncthreads();
      krem = S.s_eq_take;
      simple = (S.s_eq_take == S.s_eq_all);
      found = true;
    }
  }
  if (!found) {
    // crowded boundary (many equal or near-equal scores): exact 4-pass radix select
    uint32_t prefix = 0, mask = 0;
    krem = (uint32_t)k;
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = tid; i < 256; i += kTopkThreads) S.bins[i] = 0;
      __syncthreads();
#pragma unroll
      for (int r = 0; r < ROWS; ++r)
        if ((u[r] & mask) == prefix) atomicAdd(&S.bins[(u[r] >> shift) & 255u], 1u);
      __syncthreads();
      if (warp == 0) {
        uint32_t local = 0;
#pragma unroll
        for (int j = 0; j < 8; ++j) local += S.bins[8 * lane + j];
        uint32_t suffix = local;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t y = __shfl_down_sync(0xffffffffu, suffix, off);
          if (lane + off < 32) suffix += y;
        }
        uint32_t abv = suffix - local;
        if (abv < krem && krem <= suffix) {
          for (int j = 7; j >= 0; --j) {
            const uint32_t h = S.bins[8 * lane + j];
            if (abv + h >= krem) {
              S.s_prefix = prefix | ((uint32_t)(8 * lane + j) << shift);
              S.s_krem = krem - abv;
              break;
            }
            abv += h;
          }
        }
      }
      __syncthreads();
      prefix = S.s_prefix;
      krem = S.s_krem;
      mask |= 0xFFu << shift;
    }
    tau = prefix;
    simple = false;
  }

  return RowsThreshold{tau, krem, simple};
}

// Ascending compaction of the kept items (warp ballots, a block scan, the writes), then the
// sinks, the recent window and the padding: the token-level output.
template <int ROWS>
__device__ __forceinline__ void rows_compact_tokens(TopkRowsSmem& S, const uint32_t (&u)[ROWS], RowsThreshold th,
                                                    const TopkParams& p, int unit, int lo, int hi, int32_t* out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int w0 = warp * ROWS * 32;
  const uint32_t tau = th.tau, krem = th.krem;
  const bool simple = th.simple;
  // ---- ascending compaction: warp ballots of the selected items, block scan, writes
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t eq_base = 0;
  if (!simple) {
    // items equal to tau are taken in position order: count those before this warp's items
    uint32_t eqc = 0;
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
      eqc += __popc(__ballot_sync(0xffffffffu, u[r] == tau));
    if (lane == 0) S.wsum[warp] = eqc;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = S.wsum[lane];
      uint32_t c = w;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
        if (lane >= off) c += z;
      }
      S.wsum[lane] = c - w;
    }
    __syncthreads();
    eq_base = S.wsum[warp];
    __syncthreads();
  }
  uint32_t masks[ROWS];
  uint32_t cnt = 0, eq_run = eq_base;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    bool sel = u[r] > tau;
    const bool eq = u[r] == tau;
    if (simple) {
      sel |= eq;
    } else {
      const uint32_t be = __ballot_sync(0xffffffffu, eq);
      if (eq) sel = eq_run + __popc(be & lt) < krem;
      eq_run += __popc(be);
    }
    masks[r] = __ballot_sync(0xffffffffu, sel);
    cnt += __popc(masks[r]);
  }
  if (lane == 0) S.wsum[warp] = cnt;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = S.wsum[lane];
    uint32_t c = w;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t z = __shfl_up_sync(0xffffffffu, c, off);
      if (lane >= off) c += z;
    }
    S.wsum[lane] = c - w;
    if (lane == 31) S.s_total = c;
  }
  __syncthreads();
  uint32_t base = (uint32_t)lo + S.wsum[warp];
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const uint32_t mk = masks[r];
    if (mk == 0u) continue;                        // warp-uniform: most rows hold no kept item
    if ((mk >> lane) & 1u) out[base + __popc(mk & lt)] = lo + w0 + 32 * r + lane;
    base += __popc(mk);
  }
  const int n_chosen = (int)S.s_total;
  const int count = lo + n_chosen + p.n_recent;
  for (int i = tid; i < lo; i += kTopkThreads) out[i] = i;
  for (int i = tid; i < p.n_recent; i += kTopkThreads) out[lo + n_chosen + i] = hi + i;
  for (int i = count + tid; i < p.budget; i += kTopkThreads) out[i] = -1;
  if (tid == 0) p.count_out[unit] = count;
}

// Token-level selection with every score held in registers (up to 16 per thread), the count
// a template parameter so every pass is straight-line code.  Needs 0 < k < n <= ROWS * kTopkThreads.
template <int ROWS>
__global__ void __launch_bounds__(kTopkThreads, 1) topk_rows_kernel(const TopkParams p) {
  __shared__ TopkRowsSmem S;
  // the unit's scores on their way into L2 while the score kernel finishes (its K stream
  // has pushed the early ones out to DRAM by now)
  prefetch_lines_l2(p.score + (size_t)blockIdx.x * p.n_mid_pad, (size_t)p.n_mid_pad * 4, threadIdx.x, kTopkThreads);
  grid_dependency_wait();
  allow_dependent_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = blockIdx.x;
  const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 ? p.status : nullptr);
  int32_t* out = p.idx_out + (size_t)unit * p.budget;
  if (topk_keep_all(p, unit, t_u, out, tid, kTopkThreads)) return;
  const int lo = p.n_sink, hi = t_u - p.n_recent, n = hi - lo;
  const int k = p.budget - p.n_sink - p.n_recent;
  const float* sc = p.score + (size_t)unit * p.n_mid_pad;
  const int w0 = warp * ROWS * 32;
  uint32_t u[ROWS];
  float lmin = INFINITY, lmax = -INFINITY;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const int i = w0 + 32 * r + lane;
    const float v = i < n ? __ldcg(sc + i) : 0.f;
    u[r] = __float_as_uint(v);
    lmin = fminf(lmin, v);
    lmax = fmaxf(lmax, v);
  }
  rows_compact_tokens<ROWS>(S, u, rows_threshold<ROWS>(S, u, lmin, lmax, k), p, unit, lo, hi, out);
}

// Chunk-level selection (chunk = s > 1, the paper's policy) with every chunk's score in
// registers.  Chunk c covers positions [c s, c s + s) clipped to the middle [lo, hi), so the
// first and the last may hold fewer, and scores the sum of its members' scores in position
// order; the top k = floor(free / s) chunks (ties to the lower chunk) by rows_threshold are
// written member by member in position order.  Items are the chunks, n_items <= ROWS *
// kTopkThreads; a unit with no chunk to rank keeps all of them or none.
template <int ROWS>
__global__ void __launch_bounds__(kTopkThreads, 1) topk_rows_chunk_kernel(const TopkParams p) {
  __shared__ TopkRowsSmem S;
  prefetch_lines_l2(p.score + (size_t)blockIdx.x * p.n_mid_pad, (size_t)p.n_mid_pad * 4, threadIdx.x, kTopkThreads);
  grid_dependency_wait();
  allow_dependent_launch();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int unit = blockIdx.x;
  const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 ? p.status : nullptr);
  int32_t* out = p.idx_out + (size_t)unit * p.budget;
  if (topk_keep_all(p, unit, t_u, out, tid, kTopkThreads)) return;
  const int lo = p.n_sink, hi = t_u - p.n_recent, s = p.chunk;
  const int c_first = lo / s;
  const int n_items = hi > lo ? (hi - 1) / s - c_first + 1 : 0;
  const int k = min((p.budget - p.n_sink - p.n_recent) / s, n_items);
  const bool take_all = k >= n_items, ranked = k > 0 && !take_all;
  const float* sc = p.score + (size_t)unit * p.n_mid_pad;
  const int w0 = warp * ROWS * 32;
  auto members = [&](int i, int& a, int& b) {
    const int c = c_first + i;
    a = max(c * s, lo);
    b = min(c * s + s, hi);
  };

  // ---- chunk scores: members summed in position order, their loads eight at a time (four
  // rows' chunks in flight together; the zeros past b add nothing to scores >= +0)
  constexpr int RB = ROWS < 4 ? ROWS : 4;
  uint32_t u[ROWS];
  float lmin = INFINITY, lmax = -INFINITY;
#pragma unroll
  for (int r0 = 0; r0 < ROWS; r0 += RB) {
    int ma[RB], mb[RB];
    float v[RB];
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      const int i = w0 + 32 * (r0 + r) + lane;
      ma[r] = 0;
      mb[r] = 0;
      if (i < n_items) members(i, ma[r], mb[r]);
      v[r] = 0.f;
    }
    for (int q0 = 0; q0 < s; q0 += 8) {
      float t[RB][8];
#pragma unroll
      for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int q = ma[r] + q0 + j;
          t[r][j] = q < mb[r] ? __ldcg(sc + (q - lo)) : 0.f;
        }
#pragma unroll
      for (int r = 0; r < RB; ++r)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[r] += t[r][j];
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      u[r0 + r] = __float_as_uint(v[r]);            // +0 past n_items
      lmin = fminf(lmin, v[r]);
      lmax = fmaxf(lmax, v[r]);
    }
  }
  RowsThreshold th{0u, 0u, true};
  if (ranked) th = rows_threshold<ROWS>(S, u, lmin, lmax, k);

  // ---- kept chunks, their members in position order
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t eq_base = 0;
  if (ranked && !th.simple) {   // chunks equal to tau are taken in chunk order: those before this warp
    uint32_t eqc = 0;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) eqc += __popc(__ballot_sync(0xffffffffu, w0 + 32 * r + lane < n_items && u[r] == th.tau));
    if (lane == 0) S.wsum[warp] = eqc;
    __syncthreads();
    eq_base = __reduce_add_sync(0xffffffffu, lane < warp ? S.wsum[lane] : 0u);
    __syncthreads();
  }
  bool sel[ROWS];
  int incl[ROWS], rowoff[ROWS];
  int warp_pos = 0;
  uint32_t eq_run = eq_base;
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    const bool real = w0 + 32 * r + lane < n_items;
    bool sl = real && (take_all || (ranked && u[r] > th.tau));
    const bool eq = real && ranked && u[r] == th.tau;
    const uint32_t be = __ballot_sync(0xffffffffu, eq);
    if (eq) sl = th.simple || eq_run + __popc(be & lt) < th.krem;
    eq_run += __popc(be);
    sel[r] = sl;
    int a = 0, b = 0;
    if (real) members(w0 + 32 * r + lane, a, b);
    const int m = sl ? b - a : 0;
    int c = m;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, c, off);
      if (lane >= off) c += y;
    }
    incl[r] = c;
    rowoff[r] = warp_pos;
    warp_pos += __shfl_sync(0xffffffffu, c, 31);
  }
  if (lane == 0) S.wpos[warp] = (uint32_t)warp_pos;
  __syncthreads();
  const int base = lo + (int)__reduce_add_sync(0xffffffffu, lane < warp ? S.wpos[lane] : 0u);
  const int n_chosen = (int)__reduce_add_sync(0xffffffffu, S.wpos[lane]);
#pragma unroll
  for (int r = 0; r < ROWS; ++r) {
    if (sel[r]) {
      int a, b;
      members(w0 + 32 * r + lane, a, b);
      int o = base + rowoff[r] + incl[r] - (b - a);
      for (int q = a; q < b; ++q) out[o++] = q;
    }
  }
  const int count = lo + n_chosen + p.n_recent;
  for (int i = tid; i < lo; i += kTopkThreads) out[i] = i;
  for (int i = tid; i < p.n_recent; i += kTopkThreads) out[lo + n_chosen + i] = hi + i;
  for (int i = count + tid; i < p.budget; i += kTopkThreads) out[i] = -1;
  if (tid == 0) p.count_out[unit] = count;
}

// ============================================================================ host side

namespace {
struct ScoreKernel {
  void* fn;
  int stages, nqb;
};
// Two window-query buffers (a unit switch inside a CTA's range does not stall) and four
// K stages when they fit, else one Q buffer and as many stages as fit (measured: a fifth
// stage does not speed the kernel up).
ScoreKernel score_fn(int d, int nq_pad, bool ragged) {
  const size_t qbytes = (size_t)nq_pad * d * 2;
  const size_t kt = (size_t)kSKeys * d * 2;
  const size_t budget = 227 * 1024 - 1024 - kSQOffset;
  int stages = 4, nqb = 2;
  if (2 * qbytes + 4 * kt > budget) {
    nqb = 1;
    if (qbytes + 5 * kt <= budget) stages = 5;
  }
#define BD_SK(DD, ST, NB)                                                                              \
  if (d == DD && stages == ST && nqb == NB)                                                              \
    return {ragged ? reinterpret_cast<void*>(&score_kernel<DD, ST, NB, true>)                            \
                   : reinterpret_cast<void*>(&score_kernel<DD, ST, NB, false>), ST, NB};
  BD_SK(64, 5, 1) BD_SK(64, 4, 2) BD_SK(64, 4, 1) BD_SK(128, 5, 1) BD_SK(128, 4, 2) BD_SK(128, 4, 1)
#undef BD_SK
  return {nullptr, 0, 0};
}

uint32_t pow2_at_least(uint32_t x) {
  uint32_t r = 32;
  while (r < x) r <<= 1;
  return r;
}
}  // namespace

bool lse_plan(const bd_shape& s, int window, LsePlan* plan) {
  *plan = LsePlan{};
  const long rows = (long)(s.h_q / s.h_kv) * window;
  if (rows > 128) return false;
  const long units = (long)s.batch * s.h_kv;
  const int tpu = (s.t_ctx + kSKeys - 1) / kSKeys;
  const long total = units * tpu;
  if (total >= (1L << 31)) return false;
  int grid = (int)std::max<long>(1, std::min<long>(total, current_sm_count()));
  int tpc = (int)((total + grid - 1) / grid);
  int max_seg = 1;
  if (s.seq_lens) {
    // the lengths are read on the device: every SM gets a CTA, and the range per CTA is
    // bounded below so that a unit of tpu tiles spans at most max_seg ranges
    grid = current_sm_count();
    max_seg = (int)std::min<long>(kLMaxSeg, std::max<long>(kLMinSeg, (long)kLMaxSeg * grid / units));
    tpc = (tpu + max_seg - 2) / (max_seg - 1);
  } else {
    grid = (int)((total + tpc - 1) / tpc);
    for (long u = 0; u < std::min<long>(units, tpc); ++u)   // (the offsets repeat after tpc units)
      max_seg = std::max(max_seg, (int)((u * tpu + tpu - 1) / tpc - (u * tpu) / tpc + 1));
  }
  plan->nq_rows = (int)rows;
  plan->tiles_per_unit = tpu;
  plan->total_tiles = (int)total;
  plan->tiles_per_cta = tpc;
  plan->grid = grid;
  plan->max_seg = max_seg;
  // (at least what keeps a second CTA off the SM: it would wait for the first one's tensor memory while, with
  // the preceding kernel still on some SMs, others hold none.  A self-mode selection of 64 units of 16K, d 64:
  // 110 us with two CTAs to an SM, 76 with one.)
  const size_t smem = 2048 + (size_t)2 * 128 * s.head_dim * 2 + (size_t)kLStages * kSKeys * s.head_dim * 2 +
                      2 * 128 * sizeof(float2) + (s.seq_lens ? align_up((size_t)(units + 1) * 4, 16) : 0);
  plan->smem_bytes = std::max<size_t>(smem, 114 * 1024);
  plan->part_bytes = max_seg > 1 ? align_up((size_t)units * max_seg * 128 * sizeof(float2), 256) : 0;
  return plan->smem_bytes <= 227 * 1024;
}

size_t lse_region_bytes(const bd_shape& s, int n_q) {
  size_t bytes = 0;
  for (int n = 1; n <= n_q; ++n) {
    if (n < n_q && (s.t_ctx + n) % kSKeys != 0) continue;   // the same tiles as the next
    LsePlan lp;
    if (lse_plan(block_context(s, n), n, &lp)) bytes = std::max(bytes, lp.part_bytes);
  }
  return bytes;
}

// As many copies of a unit's rows as the 128-row operand holds, of 1, 2 and 4 (see window_lse_kernel).
static int lse_copies(int nq_rows) { return nq_rows <= 32 ? 4 : nq_rows <= 64 ? 2 : 1; }

cudaError_t launch_lse(const bd_shape& s, const LsePlan& plan, const void* k_cache, const void* q, int window,
                       int len_offset, bool window_ready, float* lse_out, void* part, int* counters, int* status,
                       cudaStream_t stream) {
  const int units = s.batch * s.h_kv;
  CUtensorMap kmap, qmap;
  cudaError_t err = make_cache_map(&kmap, k_cache, units, s.t_cap, s.t_ctx, s.head_dim, kSKeys);
  if (err != cudaSuccess) return err;
  const int copies = lse_copies(plan.nq_rows);
  err = make_rows_map(&qmap, q, (long long)units * plan.nq_rows, s.head_dim, 128 / copies);
  if (err != cudaSuccess) return err;
  LseParams p;
  p.q_win = static_cast<const __nv_bfloat16*>(q);
  p.lse = lse_out;
  p.part = static_cast<float2*>(part);
  p.counters = counters;
  p.status = status;
  p.nq_rows = plan.nq_rows;
  p.window = window;
  p.t_ctx = s.t_ctx;
  p.tiles_per_unit = plan.tiles_per_unit;
  p.total_tiles = plan.total_tiles;
  p.tiles_per_cta = plan.tiles_per_cta;
  p.max_seg = plan.max_seg;
  p.window_ready = window_ready ? 1 : 0;
  p.settled = len_offset == 0 ? INT_MAX : s.t_ctx - len_offset;   // a verify block's own rows may be fresh
  p.seq_lens = s.seq_lens;
  p.len_offset = len_offset;
  p.h_kv = s.h_kv;
  p.units = units;
  p.scale_log2 = kLog2e / sqrtf((float)s.head_dim);
  void* fn = nullptr;
#define BD_LSE(DD, R, C) \
  if (s.head_dim == DD && (s.seq_lens != nullptr) == R && copies == C) fn = reinterpret_cast<void*>(&window_lse_kernel<DD, R, C>);
  BD_LSE(64, false, 1) BD_LSE(64, false, 2) BD_LSE(64, false, 4) BD_LSE(64, true, 1) BD_LSE(64, true, 2) BD_LSE(64, true, 4)
  BD_LSE(128, false, 1) BD_LSE(128, false, 2) BD_LSE(128, false, 4) BD_LSE(128, true, 1) BD_LSE(128, true, 2)
  BD_LSE(128, true, 4)
#undef BD_LSE
  err = allow_shared_memory(fn);
  if (err != cudaSuccess) return err;
  void* args[] = {&p, &kmap, &qmap};
  return launch_kernel(fn, dim3(plan.grid), dim3(kLThreads), plan.smem_bytes, stream, args, 0);
}

bool select_plan(const bd_shape& s, int window, int budget, int n_sink, int n_recent, int chunk,
                 SelectPlan* plan) {
  *plan = SelectPlan{};
  const int group = s.h_q / s.h_kv;
  const int units = s.batch * s.h_kv;
  plan->keep_all = budget >= s.t_ctx;
  plan->nq_rows = group * window;
  plan->nq_pad = (int)align_up(plan->nq_rows, 16);
  plan->n_mid = std::max(0, s.t_ctx - n_sink - n_recent);
  plan->n_mid_pad = (int)align_up(std::max(plan->n_mid, 1), 4);
  const int free = budget - n_sink - n_recent;
  plan->need_scores = !plan->keep_all && plan->n_mid > 0 && free / chunk > 0;
  if (plan->nq_pad > 256) return false;
  const ScoreKernel sk = score_fn(s.head_dim, plan->nq_pad, s.seq_lens != nullptr);
  if (!sk.fn) return false;
  plan->tiles_per_unit = (plan->n_mid + kSKeys - 1) / kSKeys;
  plan->total_tiles = plan->tiles_per_unit * units;
  plan->grid = std::max(1, std::min(plan->total_tiles, current_sm_count()));
  plan->tiles_per_cta = (plan->total_tiles + plan->grid - 1) / plan->grid;
  plan->grid = std::max(1, (plan->total_tiles + plan->tiles_per_cta - 1) / plan->tiles_per_cta);
  plan->stages = sk.stages;
  plan->nqb = sk.nqb;
  const uint32_t acc_stride = (uint32_t)align_up(plan->nq_pad, 32);
  plan->n_acc = 4u * acc_stride <= 512u ? 4 : 2;
  plan->tmem_cols = pow2_at_least((uint32_t)plan->n_acc * acc_stride);
  plan->smem_bytes = 1024 + kSQOffset + (size_t)sk.nqb * plan->nq_pad * s.head_dim * 2 +
                     (size_t)sk.stages * kSKeys * s.head_dim * 2;
  if (s.seq_lens) {   // the units' tile table of per-sequence lengths
    plan->smem_bytes += align_up((size_t)(units + 1) * 4, 16);
    if (plan->smem_bytes > 227 * 1024) return false;
  }
  plan->score_bytes = plan->need_scores ? align_up((size_t)units * plan->n_mid_pad * 4, 256) : 0;
  plan->lse_bytes = align_up((size_t)s.batch * s.h_q * window * 4, 256);
  plan->self_mode = lse_plan(s, window, &plan->lse);   // carry mode does not need it
  return true;
}

size_t select_region_bytes(const bd_shape&, const SelectPlan& plan) {
  return plan.score_bytes + (plan.self_mode ? plan.lse_bytes + plan.lse.part_bytes : 0);
}

cudaError_t launch_select(const bd_shape& s, const SelectPlan& plan, const void* k_cache,
                          const void* q_window, const float* window_lse, int window, int budget,
                          int n_sink, int n_recent, int chunk, unsigned flags, int32_t* idx_out, int32_t* count_out,
                          void* ws_region, int* counters, int* status, cudaStream_t stream) {
  const int units = s.batch * s.h_kv;
  uint8_t* region = static_cast<uint8_t*>(ws_region);
  float* score = reinterpret_cast<float*>(region);
  cudaError_t err;
  if (plan.need_scores) {
    const float* lse = window_lse;
    if (lse == nullptr) {   // self mode: window LSE over [0, p_w]
      float* lse_buf = reinterpret_cast<float*>(region + plan.score_bytes);
      err = launch_lse(s, plan.lse, k_cache, q_window, window, 0, (flags & BD_SELECT_WINDOW_READY) != 0, lse_buf,
                       region + plan.score_bytes + plan.lse_bytes, counters, status, stream);
      if (err != cudaSuccess) return err;
      lse = lse_buf;
    }
    CUtensorMap kmap, qmap;
    err = make_cache_map(&kmap, k_cache, units, s.t_cap, s.t_ctx, s.head_dim, kSKeys);
    if (err != cudaSuccess) return err;
    err = make_rows_map(&qmap, q_window, (long long)units * plan.nq_rows, s.head_dim, plan.nq_pad);
    if (err != cudaSuccess) return err;
    ScoreParams p;
    p.q_win = static_cast<const __nv_bfloat16*>(q_window);
    p.lse_win = lse;
    p.score = score;
    p.status = status;
    p.nq_rows = plan.nq_rows;
    p.nq_pad = plan.nq_pad;
    p.window = window;
    p.t_ctx = s.t_ctx;
    p.n_sink = n_sink;
    p.mid_end = s.t_ctx - n_recent;
    p.n_mid_pad = plan.n_mid_pad;
    p.tiles_per_unit = plan.tiles_per_unit;
    p.total_tiles = plan.total_tiles;
    p.tiles_per_cta = plan.tiles_per_cta;
    p.acc_stride = (int)align_up(plan.nq_pad, 32);
    p.n_acc = plan.n_acc;
    p.tmem_cols = plan.tmem_cols;
    p.scale_log2 = kLog2e / sqrtf((float)s.head_dim);
    p.seq_lens = s.seq_lens;
    p.h_kv = s.h_kv;
    p.window_ready = (flags & BD_SELECT_WINDOW_READY) ? 1 : 0;
    void* fn = score_fn(s.head_dim, plan.nq_pad, s.seq_lens != nullptr).fn;
    err = allow_shared_memory(fn);
    if (err != cudaSuccess) return err;
    void* args[] = {&p, &kmap, &qmap};
    err = launch_kernel(fn, dim3(plan.grid), dim3(kSThreads), plan.smem_bytes, stream, args, 0);
    if (err != cudaSuccess) return err;
  }
  TopkParams tp;
  tp.score = score;
  tp.idx_out = idx_out;
  tp.count_out = count_out;
  tp.t_ctx = s.t_ctx;
  tp.budget = budget;
  tp.n_sink = n_sink;
  tp.n_recent = n_recent;
  tp.chunk = chunk;
  tp.n_mid_pad = plan.n_mid_pad;
  tp.keep_all = plan.keep_all ? 1 : 0;
  tp.seq_lens = s.seq_lens;
  tp.h_kv = s.h_kv;
  tp.status = status;
  void* targs[] = {&tp};
  const int free = budget - n_sink - n_recent;
  if (!plan.keep_all && plan.need_scores && chunk == 1 && free < plan.n_mid && plan.n_mid <= 16 * kTopkThreads) {
    const int rows = (plan.n_mid + kTopkThreads - 1) / kTopkThreads;
    void* fn = rows <= 1   ? reinterpret_cast<void*>(&topk_rows_kernel<1>)
               : rows <= 2 ? reinterpret_cast<void*>(&topk_rows_kernel<2>)
               : rows <= 4 ? reinterpret_cast<void*>(&topk_rows_kernel<4>)
               : rows <= 8 ? reinterpret_cast<void*>(&topk_rows_kernel<8>)
                           : reinterpret_cast<void*>(&topk_rows_kernel<16>);
    return launch_kernel(fn, dim3(units), dim3(kTopkThreads), 0, stream, targs, 0);
  }
  // One CTA per unit while it holds the items and the batch fills the GPU that way; a
  // cluster per unit (bd_topk_long.cu) where a unit is too long for that, or where SMs are
  // left: token level from four CTAs a unit on (a select call of 8 units of 32K positions 29.6
  // us with one CTA, 26.8 in the cluster; 64 units 107.7 against 107.9, 128 units 195.6 against
  // 210.3), chunk level, whose member sums cost more, from two on (chunks of 8: 24 units of 36K
  // 58.7 against 53.7 us, 128 units of 20K 128.7 against 140.3; of 16K, 8 units 16.8 against 18.3).
  int n_items = plan.n_mid;
  const long sms = current_sm_count();
  if (!plan.keep_all && plan.need_scores && chunk == 1 && plan.n_mid <= kLeanMaxItems && 4L * units > sms) {
    const size_t smem = (size_t)align_up(plan.n_mid, 4) * 4;
    void* fn = reinterpret_cast<void*>(&topk_token_kernel);
    err = allow_shared_memory(fn, 64 * 1024);   // (its own arrays: 34 KB)
    if (err != cudaSuccess) return err;
    return launch_kernel(fn, dim3(units), dim3(kTopkThreads), smem, stream, targs, 0);
  }
  if (!plan.keep_all && plan.need_scores && chunk > 1) {
    const int lo = n_sink, hi = s.t_ctx - n_recent;
    n_items = hi > lo ? (hi - 1) / chunk - lo / chunk + 1 : 0;
    if (n_items <= 16 * kTopkThreads && (plan.n_mid <= 16 * kTopkThreads || 2L * units > sms)) {
      const int rows = std::max(1, (n_items + kTopkThreads - 1) / kTopkThreads);
      void* fn = rows <= 1   ? reinterpret_cast<void*>(&topk_rows_chunk_kernel<1>)
                 : rows <= 2 ? reinterpret_cast<void*>(&topk_rows_chunk_kernel<2>)
                 : rows <= 4 ? reinterpret_cast<void*>(&topk_rows_chunk_kernel<4>)
                 : rows <= 8 ? reinterpret_cast<void*>(&topk_rows_chunk_kernel<8>)
                             : reinterpret_cast<void*>(&topk_rows_chunk_kernel<16>);
      return launch_kernel(fn, dim3(units), dim3(kTopkThreads), 0, stream, targs, 0);
    }
  }
  return plan.keep_all || !plan.need_scores ? launch_topk_plain(tp, units, stream)
                                            : launch_topk_long(tp, units, n_items, stream);
}

}  // namespace bd
