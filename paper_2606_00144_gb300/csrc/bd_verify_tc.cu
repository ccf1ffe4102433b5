// Verifier block attention with many query rows per KV head (long drafts, wide GQA groups) on
// the 5th-generation tensor cores.  Same result and stream-K cut as verify_kernel
// (bd_verify.cu), whose mma.sync sub-tiles are bound by the tensor pipe beyond a few n8 tiles.
//
//   S = Q K^T       M = 128 query rows (TMEM lanes, padded), N = 128 keys, K = D; both operands in
//                   shared memory by TMA;
//   P = exp2(S - m) one thread per row, in two bf16 terms P_hi + P_lo (as in bd_attn_warp.cuh),
//                   written over S in TMEM;
//   O += P V        A = P_hi, then P_lo, from TMEM; B = the V tile as it lies in shared memory (keys x D,
//                   MN-major), O in TMEM.
//
// A job is one (128-key tile, M tile) pair.  Jobs alternate between two S/P buffers, two O
// accumulators and two groups of four softmax warps: with one M tile (up to 128 rows) the groups
// take alternate key tiles and their halves meet at the end of a segment; with two (up to 256 rows)
// each group owns an M tile and both read the same K and V stages, so K and V are read once.
//   warp 0      producer: K and V tiles through one ring, in the order the MMAs use them;
//   warp 1      MMA issuer: S of job j before P V of job j - 1, so a softmax overlaps the MMAs;
//   warps 2-9   softmax, and the segment's output.
// Bound by HBM up to 128 rows (64 units of 16K keys, 84 rows: 89.1 us, 6.0 TB/s; verify_kernel took
// 313.8 us), by the tensor pipe with two M tiles (16 units of 16K, 168 rows: 45 us, of which the MMAs
// of a CTA's 28 jobs take 26; verify_kernel, in two chunks, 160 us).
// The running max may trail the true one by 2^8: O is rescaled in TMEM only when a row's max
// grows by more, which after a segment's first tiles is rare.
// Every segment of a unit that spans CTAs is written as a partial, four columns of all rows at a
// time ([D/4][rows] float4: a warp of row threads writes 512 contiguous bytes; row-major partials
// took 3 us to write), and verify_tc_merge_kernel merges.
#include "bd_common.cuh"
#include "bd_internal.h"
#include "bd_verify.cuh"

namespace bd {

constexpr int kTSoftmax = 256;                       // softmax threads
constexpr float kTSlack = 8.f;                       // log2 of how far the running max may trail
constexpr uint32_t kTHalf = kVTcKeys * 128;          // one 64-column half of a 128-row tile
constexpr size_t kTFixed = 1024 + 1024 + 2 * 128 * sizeof(float2);   // alignment, barriers, (m, l) exchange

template <int D, int NQT>
struct VerifyTcSmem {
  static constexpr uint32_t TILE = kVTcKeys * D * 2;   // a K, V or Q tile
  // K and V tiles in flight: what 227 KB hold beside the queries and the units' table
  static constexpr int SLOTS = D == 64 ? 8 : (NQT == 1 ? 5 : 4);
  static constexpr size_t kTotal = kTFixed + (size_t)(NQT + SLOTS) * TILE;
};

// Rows [r0, 128) of a V tile in shared memory become zero, by one warp, before that warp's MMAs read them.
// With per-sequence lengths the last tile of a sequence shorter than the longest one reaches cache rows
// past its own block, which nobody has promised to be finite, and a weight of 0 times NaN is NaN.
template <int D>
__device__ __forceinline__ void clear_rows(uint8_t* tile, int r0, int lane) {
  if (r0 >= kVTcKeys) return;
  constexpr int CH = D / 8, PER = 32 / CH;          // 16-byte chunks of a row; rows at a time
  const int c = lane % CH;
  uint8_t* at = tile + c / 8 * kTHalf + c % 8 * 16;
#pragma unroll 1
  for (int r = r0 + lane / CH; r < kVTcKeys; r += PER) *reinterpret_cast<uint4*>(at + r * 128) = make_uint4(0u, 0u, 0u, 0u);
  fence_proxy_async_smem();
  __syncwarp();
}

// UNIFORM: one shared context length; the other instance lays out per-sequence lengths.
template <int D, int NQT, bool UNIFORM>
__global__ void __launch_bounds__(kVTcThreads, 1) verify_tc_kernel(const VerifyParams p,
                                                                 const __grid_constant__ CUtensorMap kmap,
                                                                 const __grid_constant__ CUtensorMap vmap,
                                                                 const __grid_constant__ CUtensorMap qmap) {
  using L = VerifyTcSmem<D, NQT>;
  constexpr int SLOTS = L::SLOTS;
  constexpr uint32_t TILE = L::TILE;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem);   // [SLOTS] the ring
  uint64_t* empty_bar = full_bar + SLOTS;
  uint64_t* s_full = empty_bar + SLOTS;                     // [2] scores of buffer b are in TMEM
  uint64_t* p_ready = s_full + 2;                           // [2] the weights of buffer b are in TMEM
  uint64_t* pv_done = p_ready + 2;                          // [2] buffer b is free, O[b] up to date
  uint64_t* q_full = pv_done + 2;
  uint64_t* q_empty = q_full + 1;
  uint64_t* o_free = q_empty + 1;                           // the segment's O has been read
  uint64_t* drain_bar = o_free + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* live_s = reinterpret_cast<int*>(tmem_slot + 2);      // [SLOTS] per-sequence lengths: the block's rows in a segment's last V tile
  float2* ml_s = reinterpret_cast<float2*>(smem + 1024);    // [2][128] (m, l) of the two groups
  uint8_t* qbuf = smem + 1024 + 2 * 128 * sizeof(float2);   // NQT x TILE
  uint8_t* ring = qbuf + NQT * TILE;                        // SLOTS x TILE
  int* pref = reinterpret_cast<int*>(ring + SLOTS * TILE);  // per-sequence lengths: [units + 1]

  const int tid = threadIdx.x, warp = uniform_warp(), lane = tid & 31;
  VerifyMap map{nullptr, p.tiles_per_unit, p.seg_cost, p.units, p.vtiles_per_cta};
  if (!UNIFORM) {
    grid_dependency_wait();
    lay_out_units<kVTcThreads, kVTcKeys>(p, p.units, reinterpret_cast<int*>(smem + 512), pref);
    map.pref = pref;
    map.vtpc = max((pref[p.units] + (int)gridDim.x - 1) / (int)gridDim.x, p.vtiles_per_cta);
  }
  const int v_total = map.vbase(p.units);
  const int v0 = min(v_total, (int)blockIdx.x * map.vtpc), v1 = min(v_total, v0 + map.vtpc);
  if (v0 >= v1) return;                           // whole CTA idle
  const int u_first = map.unit_of(v0), u_last = map.unit_of(v1 - 1);

  if (tid == 0) {
    for (int s = 0; s < SLOTS; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&s_full[b], 1);
      mbar_init(&p_ready[b], 4);
      mbar_init(&pv_done[b], 1);
    }
    mbar_init(q_full, 1);
    mbar_init(q_empty, 1);
    mbar_init(o_free, 8);
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // S/P buffer b: columns 128 b; O[b]: columns 256 + D b

  // Ring position of a segment's tiles, n of them, relative to its first: the order the MMAs
  // use them in, K0 K1 V0 K2 V1 ... V(n-1).
  auto k_pos = [](int i) { return i == 0 ? 0 : 2 * i - 1; };
  auto v_pos = [](int i, int n) { return i == n - 1 ? 2 * n - 1 : 2 * i + 2; };

  // A unit's queries (rows past the M tile's own are computed and discarded).  The first
  // segment's are requested by a softmax warp once the dependency wait is over, among the first K
  // and V tiles: context rows are older than the preceding kernel, the queries may not be, and
  // behind a full ring of tiles they arrived 2 us later.  Later segments' by the producer.
  auto load_q = [&](int unit) {
    const int kv_unit = unit / p.row_chunks;
    const int row0 = kv_unit * p.rows_total + (unit - kv_unit * p.row_chunks) * p.nq_rows;
    mbar_arrive_expect_tx(q_full, NQT * TILE);
#pragma unroll
    for (int qt = 0; qt < NQT; ++qt)
#pragma unroll
      for (int h = 0; h < D / 64; ++h)
        tma_load_2d(qbuf + qt * TILE + h * kTHalf, &qmap, q_full, 64 * h, row0 + qt * p.tile_rows);
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    allow_dependent_launch();
    if (lane == 0) {
      tma_prefetch_map(&kmap);
      tma_prefetch_map(&vmap);
      tma_prefetch_map(&qmap);
      bool ok = true, waited = !UNIFORM;
      int issued = 0, seg = 0;                      // ring position; segments begun
      for (int unit = u_first; unit <= u_last && ok; ++unit) {
        const int tb = map.first_tile(unit, v0), te = map.end_tile(unit, v1), n = te - tb;
        if (n <= 0) continue;
        const int kv_unit = unit / p.row_chunks;
        const int t_unit = UNIFORM ? 0 : p.seq_lens[kv_unit / p.h_kv];   // (on its way; used at the segment's end)
        // entry i of the segment: K of tile 0 or (odd i) of tile (i + 1) / 2, else V
        auto entry_tile = [&](int i) { return i == 0 ? 0 : i == 2 * n - 1 ? n - 1 : (i & 1) ? (i + 1) >> 1 : (i >> 1) - 1; };
        auto issue = [&](int i) {
          const int s = issued % SLOTS;
          if (issued >= SLOTS) ok = mbar_wait(&empty_bar[s], ((issued / SLOTS) & 1) ^ 1, p.status, abort_flag);
          if (!ok) return;
          const int key0 = (tb + entry_tile(i)) * kVTcKeys;
          if (!waited && key0 + kVTcKeys > p.t_ctx) {   // this tile holds rows of the block itself
            grid_dependency_wait();
            waited = true;
          }
          const CUtensorMap* m = i == 0 || ((i & 1) && i != 2 * n - 1) ? &kmap : &vmap;
          if (!UNIFORM && i == 2 * n - 1) live_s[s] = min(max(t_unit, 1), p.t_ctx) + p.n_q - key0;
          mbar_arrive_expect_tx(&full_bar[s], TILE);
#pragma unroll
          for (int h = 0; h < D / 64; ++h) tma_load_3d(ring + s * TILE + h * kTHalf, m, &full_bar[s], 64 * h, key0, kv_unit);
          ++issued;
        };
        // a later segment's first entries stream while its predecessor's last scores still read
        // the query tile (their slots depend on that segment alone)
        const int pre = seg == 0 ? 0 : min(2 * n, SLOTS - 1);
        for (int i = 0; i < pre && ok; ++i) issue(i);
        if (ok && seg > 0) {
          ok = mbar_wait(q_empty, (seg - 1) & 1, p.status, abort_flag);
          if (ok) load_q(unit);
        }
        if (!ok) break;
        ++seg;
        for (int i = pre; i < 2 * n && ok; ++i) issue(i);
      }
      if (*abort_flag) {   // no copy may land in shared memory after the CTA exits
        for (int t = max(0, issued - SLOTS); t < issued; ++t)
          mbar_wait(&full_bar[t % SLOTS], (t / SLOTS) & 1, p.status, nullptr);
        if (seg > 0) mbar_wait(q_full, (seg - 1) & 1, p.status, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer (whole warp, see tc_mma_ss)
    allow_dependent_launch();
    const uint32_t lead = elect_leader();
    constexpr uint32_t idesc_s = umma_idesc_bf16(128, kVTcKeys);
    constexpr uint32_t idesc_o = umma_idesc_bf16(128, D) | kIdescBMnMajor;
    bool ok = true;
    int jg = 0, base = 0, seg = 0;                  // jobs, ring position and segments before this one
    for (int unit = u_first; unit <= u_last && ok; ++unit) {
      const int tb = map.first_tile(unit, v0), te = map.end_tile(unit, v1), n = te - tb;
      if (n <= 0) continue;
      const int nj = n * NQT;
      if (!mbar_wait_warp(q_full, seg & 1, p.status, abort_flag)) break;
      for (int j = 0; j <= nj; ++j) {
        if (j < nj) {                               // S of job j
          const int b = (jg + j) & 1, i = j / NQT, qt = j % NQT;
          const int r = base + k_pos(i), s = r % SLOTS;
          // the buffer's previous weights have been used
          if (jg + j >= 2) ok = mbar_wait_warp(&pv_done[b], (((jg + j) >> 1) - 1) & 1, p.status, abort_flag);
          if (ok && qt == 0) ok = mbar_wait_warp(&full_bar[s], (r / SLOTS) & 1, p.status, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t a_lo = desc_k(smem_u32(qbuf + qt * TILE));
          const uint32_t b_lo = desc_k(smem_u32(ring + s * TILE));
#pragma unroll
          for (int ks = 0; ks < D / 16; ++ks) {
            const uint32_t off = ((ks >> 2) * kTHalf + (ks & 3) * 32) / 16;
            tc_mma_ss(lead, tmem_base + 128 * b, a_lo + off, b_lo + off, idesc_s, ks > 0 ? 1u : 0u);
          }
          tc_commit(lead, &s_full[b]);
          if (qt == NQT - 1) tc_commit(lead, &empty_bar[s]);
          if (j == nj - 1) tc_commit(lead, q_empty);
        }
        if (j > 0) {                                // P V of job j - 1
          const int jj = jg + j - 1, b = jj & 1, i = (j - 1) / NQT, qt = (j - 1) % NQT;
          const int r = base + v_pos(i, n), s = r % SLOTS;
          if (j == 1 && seg > 0) ok = mbar_wait_warp(o_free, (seg - 1) & 1, p.status, abort_flag);
          if (ok && qt == 0) ok = mbar_wait_warp(&full_bar[s], (r / SLOTS) & 1, p.status, abort_flag);
          if (!UNIFORM && ok && i == n - 1 && qt == 0) clear_rows<D>(ring + s * TILE, live_s[s], lane);
          if (ok) ok = mbar_wait_warp(&p_ready[b], (jj >> 1) & 1, p.status, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t v_lo = desc_mn(smem_u32(ring + s * TILE), kTHalf);
          const uint32_t d_tmem = tmem_base + 256 + D * b, a_tmem = tmem_base + 128 * b;
          const uint32_t first = j - 1 < 2 ? 0u : 1u;   // O[b]'s first job of the segment
#pragma unroll 1
          for (int t = 0; t < 2; ++t)                // P_hi, then P_lo
#pragma unroll
            for (int ks = 0; ks < kVTcKeys / 16; ++ks)
              tc_mma_ts(lead, d_tmem, a_tmem + 32 * (ks >> 1) + 8 * (ks & 1) + 16 * t, v_lo + ks * (16 * 128 / 16), idesc_o,
                        t + ks > 0 ? 1u : first);
          tc_commit(lead, &pv_done[b]);
          if (qt == NQT - 1) tc_commit(lead, &empty_bar[s]);
        }
      }
      jg += nj;
      base += 2 * n;
      ++seg;
    }
    // every MMA this warp issued has completed before TMEM is released
    tc_commit(lead, drain_bar);
    mbar_wait(drain_bar, 0, p.status, nullptr);
  } else {
    // ---------------------------------------------------------------- softmax: one query row per thread
    if (UNIFORM) grid_dependency_wait();           // the queries come from the preceding kernels
    if (warp == 2) {
      int unit = u_first;
      while (unit <= u_last && map.first_tile(unit, v0) >= map.end_tile(unit, v1)) ++unit;
      if (unit <= u_last && lane == 0) load_q(unit);
      __syncwarp();
    }
    allow_dependent_launch();
    const int grp = (warp - 2) >> 2;               // jobs of parity grp, S/P buffer and O[grp]
    const int quad = warp & 3;                     // TMEM lanes quad*32 .. quad*32+31
    const int row = quad * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(quad * 32) << 16);
    const uint32_t t_s = t_lane + 128 * grp;
    // after a wait gives up, a warp keeps walking without touching TMEM, so that all eight
    // warps still meet at the segment ends
    bool alive = true;
    int jg = 0;
    for (int unit = u_first; unit <= u_last; ++unit) {
      const int tb = map.first_tile(unit, v0), te = map.end_tile(unit, v1), n = te - tb;
      if (n <= 0) continue;
      const int kv_unit = unit / p.row_chunks;
      const int row_base = (unit - kv_unit * p.row_chunks) * p.nq_rows;   // first row of this chunk
      const int rows = min(p.nq_rows, p.rows_total - row_base);
      const int t_unit =
          UNIFORM ? p.t_ctx : unit_context(p.seq_lens, kv_unit, p.h_kv, p.t_ctx, tid == 64 ? p.status : nullptr);
      const int m0 = NQT == 2 ? grp * p.tile_rows : 0;                    // the M tile's first row of the chunk
      const int m_rows = NQT == 2 && grp == 0 ? min(rows, p.tile_rows) : rows - m0;
      const int lim = row < m_rows ? t_unit + (row_base + m0 + row) % p.n_q : -1;   // last visible key
      const bool warp_live = quad * 32 < m_rows;
      float m = -INFINITY, l = 0.f;                // log2 units
      const int nj = n * NQT;
      for (int j = (jg + grp) & 1; j < nj; j += 2) {
        const int use = (jg + j) >> 1;             // uses of this buffer before this one
        alive = __all_sync(0xffffffffu, alive && mbar_wait(&s_full[grp], use & 1, p.status, abort_flag));
        if (!alive) continue;
        tc_fence_after();
        if (warp_live) {
          // two passes over halves of 64 keys: the second half's maximum, the first half's (its
          // scores stay in registers), the weights of the first, the second again
          const int key0 = (tb + j / NQT) * kVTcKeys;
          const bool masked = key0 + kVTcKeys - 1 > t_unit;   // some key is hidden from some row
          float v[64];
          auto load_half = [&](int h) {
            tc_ld_32cols(t_s + 64 * h, *reinterpret_cast<float(*)[32]>(&v[0]));
            tc_ld_32cols(t_s + 64 * h + 32, *reinterpret_cast<float(*)[32]>(&v[32]));
            tc_wait_ld();
            if (masked) {
#pragma unroll
              for (int c = 0; c < 64; ++c) v[c] = key0 + 64 * h + c <= lim ? v[c] : -INFINITY;
            }
          };
          auto half_max = [&]() {
            float mx[4] = {fmaxf(v[0], v[4]), fmaxf(v[1], v[5]), fmaxf(v[2], v[6]), fmaxf(v[3], v[7])};
#pragma unroll
            for (int c = 8; c < 64; c += 8)
#pragma unroll
              for (int e = 0; e < 4; ++e) mx[e] = fmaxf(mx[e], fmaxf(v[c + e], v[c + 4 + e]));
            return fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3]));
          };
          load_half(1);
          const float mx1 = half_max();
          load_half(0);
          const float mxs = fmaxf(half_max(), mx1) * p.scale_log2;
          const bool grow = mxs > m + kTSlack;     // m = -inf: any visible key
          float alpha = 1.f;
          if (grow) {
            alpha = fast_exp2(m - mxs);
            m = mxs;
            l *= alpha;
          }
          if (j >= 2 && __any_sync(0xffffffffu, grow)) {
            // O[grp] holds earlier tiles: scaled once the MMA that adds the last of them is done
            alive = __all_sync(0xffffffffu, mbar_wait(&pv_done[grp], (use - 1) & 1, p.status, abort_flag));
            if (!alive) continue;
            tc_fence_after();
#pragma unroll 1
            for (int c = 0; c < D; c += 16) {
              float o[16];
              const uint32_t t_o = t_lane + 256 + D * grp + c;
              tc_ld_16cols(t_o, o);
              tc_wait_ld();
              uint32_t ob[16];
#pragma unroll
              for (int e = 0; e < 16; ++e) ob[e] = __float_as_uint(o[e] * alpha);
              tc_st_16cols(t_o, ob);
            }
          }
          const float2 cc = make_float2(p.scale_log2, p.scale_log2);
          const float nms = m == -INFINITY ? 0.f : -m;
          const float2 nm = make_float2(nms, nms);
          float2 a0 = make_float2(0.f, 0.f), a1 = a0;
          // 32 keys' weights over their scores: columns c .. c+15 P_hi, c+16 .. c+31 P_lo
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            if (h == 1) load_half(1);
#pragma unroll
            for (int c = 0; c < 64; c += 32) {
              uint32_t hi[16], lo[16];
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                float2 x0 = ffma2(make_float2(v[c + 2 * e], v[c + 2 * e + 1]), cc, nm);
                float2 x1 = ffma2(make_float2(v[c + 2 * e + 2], v[c + 2 * e + 3]), cc, nm);
                x0 = make_float2(fast_exp2(x0.x), fast_exp2(x0.y));
                x1 = make_float2(fast_exp2(x1.x), fast_exp2(x1.y));
                a0 = fadd2(a0, x0);
                a1 = fadd2(a1, x1);
                split_bf16x2(x0.x, x0.y, hi[e], lo[e]);
                split_bf16x2(x1.x, x1.y, hi[e + 1], lo[e + 1]);
              }
              tc_st_16cols(t_s + 64 * h + c, hi);
              tc_st_16cols(t_s + 64 * h + c + 16, lo);
            }
          }
          l += (a0.x + a0.y) + (a1.x + a1.y);
          tc_wait_st();
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_ready[grp]);
      }
      // ---------------------------------------------------------------- end of the segment
      // the last job of each accumulator in this segment (none: fewer than two jobs)
      const int last = jg + nj - 1;
      const int last_own = (last & 1) == grp ? last : last - 1;
      const int last_oth = last + last - 1 - last_own;
      const bool has_own = last_own >= jg, has_oth = NQT == 1 && last_oth >= jg;
      jg += nj;
      if (has_own)
        alive = __all_sync(0xffffffffu, alive && mbar_wait(&pv_done[grp], (last_own >> 1) & 1, p.status, abort_flag));
      if (has_oth)
        alive = __all_sync(0xffffffffu, alive && mbar_wait(&pv_done[grp ^ 1], (last_oth >> 1) & 1, p.status, abort_flag));
      tc_fence_after();
      float f_own = 1.f, f_oth = 0.f, M = m, S = l;
      if (NQT == 1) {
        ml_s[grp * 128 + row] = make_float2(m, l);
        named_bar(1, kTSoftmax);
        const float2 o = ml_s[(grp ^ 1) * 128 + row];
        M = fmaxf(m, o.x);
        f_own = m == -INFINITY ? 0.f : fast_exp2(m - M);
        f_oth = o.x == -INFINITY ? 0.f : fast_exp2(o.x - M);
        S = f_own * l + f_oth * o.y;
      }
      const float inv = S > 0.f ? 1.f / S : 0.f;
      f_own *= inv;
      f_oth *= inv;
      const int c = blockIdx.x, c_first = map.owner(unit, 0), c_last = map.owner(unit, map.tiles(unit) - 1);
      const bool whole = c_first == c_last;
      if (c == c_first && tid == 64 && p.max_seg > 1) p.nseg[unit] = c_last - c_first + 1;
      const size_t pslot = (size_t)unit * p.max_seg + (c - c_first);                            // the partial
      const size_t orow = (size_t)kv_unit * p.rows_total + row_base + m0 + row;                 // output row
      if (alive && warp_live) {
        if (row < m_rows && (NQT == 2 || grp == 0)) {
          const float lse = S > 0.f ? (M + log2f(S)) * kLn2 : -INFINITY;
          if (!whole) p.lse_part[pslot * p.nq_rows + m0 + row] = lse;
          else if (p.lse) p.lse[orow] = lse;
        }
        // NQT 1: each group combines half of the columns of both accumulators
        constexpr int CW = NQT == 1 ? D / 2 : D;
        const int col0 = NQT == 1 ? grp * CW : 0;
#pragma unroll 1
        for (int cb = 0; cb < CW; cb += 16) {
          float o[16], x[16];
          if (has_own) tc_ld_16cols(t_lane + 256 + D * grp + col0 + cb, o);
          if (has_oth) tc_ld_16cols(t_lane + 256 + D * (grp ^ 1) + col0 + cb, x);
          tc_wait_ld();
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float a = has_own ? o[e] * f_own : 0.f;
            o[e] = has_oth ? fmaf(x[e], f_oth, a) : a;
          }
          if (row < m_rows) {
            if (whole) {
              uint4* dst = reinterpret_cast<uint4*>(p.o + orow * D + col0 + cb);
#pragma unroll
              for (int e = 0; e < 2; ++e)
                dst[e] = make_uint4(pack_bf16x2(o[8 * e], o[8 * e + 1]), pack_bf16x2(o[8 * e + 2], o[8 * e + 3]),
                                    pack_bf16x2(o[8 * e + 4], o[8 * e + 5]), pack_bf16x2(o[8 * e + 6], o[8 * e + 7]));
            } else {
              float4* dst = reinterpret_cast<float4*>(p.o_part) + pslot * (D / 4) * p.nq_rows +
                            (size_t)((col0 + cb) / 4) * p.nq_rows + m0 + row;
#pragma unroll
              for (int e = 0; e < 4; ++e) dst[e * p.nq_rows] = make_float4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
            }
          }
        }
      }
      // (the next segment's (m, l) are written after its P V, which waits for this barrier)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(o_free);
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, 512);
}

// Merge of the segments' partials: one CTA per (unit, eight output rows); a unit whose segment
// count is 1 was written by the verify kernel itself.  Thread (row, four columns, segment group)
// requests all of its parts at once, before the weights are known; the NG groups, as many as keep
// that to nine parts a thread, meet in shared memory.  (8 units of 84 rows and 17 parts: parts
// eight at a time in one thread made the call 3 us longer; 32 units of 104 rows and 5 parts: CTAs of two rows
// 4 us longer.)
constexpr int kTMergeRows = 8;
constexpr int kTMergePer = 9;       // parts in flight per thread
template <int D, int NG>
__global__ void __launch_bounds__(kTMergeRows* D / 4 * NG)
    verify_tc_merge_kernel(const float* o_part, const float* lse_part, const int* nseg, int max_seg, int nq,
                           int rows_total, int row_chunks, __nv_bfloat16* o, float* lse) {
  constexpr int R = kTMergeRows, PER = kTMergePer, WARPS = R * D / 4 * NG / 32;
  static_assert(4 * PER >= kVMaxSeg, "four groups hold every part");
  grid_dependency_wait();
  allow_dependent_launch();
  __shared__ float w[R][kVMaxSeg];
  __shared__ float4 sum[NG][R * D / 4];
  const int unit = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kv_unit = unit / row_chunks, row_base = (unit - kv_unit * row_chunks) * nq;
  const int rows = min(nq, rows_total - row_base), r0 = R * blockIdx.y;
  const int n = min(__ldcg(nseg + unit), kVMaxSeg);
  if (n <= 1 || r0 >= rows) return;
  const size_t base = (size_t)unit * max_seg, orow0 = (size_t)kv_unit * rows_total + row_base;
  const int item = tid % (R * D / 4), g = tid / (R * D / 4), r = r0 + item % R, q = item / R;
  const float4* part = reinterpret_cast<const float4*>(o_part) + (base * (D / 4) + q) * nq + min(r, rows - 1);
  const size_t step = (size_t)(D / 4) * nq;
  float4 v[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k)
    v[k] = g + NG * k < n ? __ldcg(part + (g + NG * k) * step) : make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = warp; i < R && r0 + i < rows; i += WARPS) {   // a row's weights exp(lse_s - L)
    const int rr = r0 + i;
    const float l0 = lane < n ? __ldcg(lse_part + (base + lane) * nq + rr) : -INFINITY;
    const float l1 = lane + 32 < n ? __ldcg(lse_part + (base + lane + 32) * nq + rr) : -INFINITY;
    float mx = fmaxf(l0, l1);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    const float e0 = mx == -INFINITY ? 0.f : fast_exp2((l0 - mx) * kLog2e);
    const float e1 = mx == -INFINITY ? 0.f : fast_exp2((l1 - mx) * kLog2e);
    float tot = e0 + e1;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, off);
    const float inv = tot > 0.f ? 1.f / tot : 0.f;
    if (lane < n) w[i][lane] = e0 * inv;
    if (lane + 32 < n) w[i][lane + 32] = e1 * inv;
    if (lane == 0 && lse) lse[orow0 + rr] = mx == -INFINITY ? -INFINITY : mx + logf(tot);
  }
  __syncthreads();
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const float wk = g + NG * k < n && r < rows ? w[item % R][g + NG * k] : 0.f;
    if (wk != 0.f) {                              // an empty part never enters the sum
      acc.x += wk * v[k].x;
      acc.y += wk * v[k].y;
      acc.z += wk * v[k].z;
      acc.w += wk * v[k].w;
    }
  }
  if (NG > 1) {
    sum[g][item] = acc;
    __syncthreads();
  }
  if (g != 0 || r >= rows) return;
#pragma unroll
  for (int h = 1; h < NG; ++h) {
    const float4 b = sum[h][item];
    acc.x += b.x;
    acc.y += b.y;
    acc.z += b.z;
    acc.w += b.w;
  }
  uint2 packed;
  packed.x = pack_bf16x2(acc.x, acc.y);
  packed.y = pack_bf16x2(acc.z, acc.w);
  *reinterpret_cast<uint2*>(o + (orow0 + r) * D + 4 * q) = packed;
}

// ============================================================================ host side

cudaError_t launch_verify_tc_merge(int head_dim, int units, const VerifyParams& p, cudaStream_t stream) {
  const float* op = p.o_part;
  const float* lp = p.lse_part;
  const int* ns = p.nseg;
  int max_seg = p.max_seg, nq = p.nq_rows, rows_total = p.rows_total, chunks = p.row_chunks;
  __nv_bfloat16* o = p.o;
  float* l = p.lse;
  void* args[] = {&op, &lp, &ns, &max_seg, &nq, &rows_total, &chunks, &o, &l};
  const int ng = max_seg <= kTMergePer ? 1 : max_seg <= 2 * kTMergePer ? 2 : 4;
  const void* fn = nullptr;
#define BD_TM(D, N) \
  if (head_dim == D && ng == N) fn = reinterpret_cast<const void*>(&verify_tc_merge_kernel<D, N>);
  BD_TM(64, 1) BD_TM(64, 2) BD_TM(64, 4) BD_TM(128, 1) BD_TM(128, 2) BD_TM(128, 4)
#undef BD_TM
  return launch_kernel(fn, dim3(units, (nq + kTMergeRows - 1) / kTMergeRows), dim3(kTMergeRows * head_dim / 4 * ng), 0,
                       stream, args, 0);
}

size_t verify_tc_smem(int head_dim, int q_tiles) {
  if (head_dim == 64) return q_tiles == 1 ? VerifyTcSmem<64, 1>::kTotal : VerifyTcSmem<64, 2>::kTotal;
  return q_tiles == 1 ? VerifyTcSmem<128, 1>::kTotal : VerifyTcSmem<128, 2>::kTotal;
}

const void* verify_tc_fn(int head_dim, int q_tiles, bool ragged) {
#define BD_VT(D, N) \
  if (head_dim == D && q_tiles == N)            \
    return ragged ? reinterpret_cast<const void*>(&verify_tc_kernel<D, N, false>) : reinterpret_cast<const void*>(&verify_tc_kernel<D, N, true>);
  BD_VT(64, 1) BD_VT(64, 2) BD_VT(128, 1) BD_VT(128, 2)
#undef BD_VT
  return nullptr;
}

}  // namespace bd
