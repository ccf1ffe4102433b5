// Top-B selection over long middles (more items than one CTA holds in registers, or few
// units): one thread-block cluster per (sequence, KV head) unit.  The CTAs of a cluster share
// the items; every step that needs the whole unit (value range, histogram, the boundary bin's
// items, the output offsets) is one exchange through distributed shared memory, after which
// each CTA derives the same threshold by itself.  What bounds it is the chain of exchanges
// (four cluster barriers) and the slowest CTA's passes over its own items.  A select call over
// 8 units of 128K positions: 377 us with one CTA per unit (scores re-read by every radix pass),
// 65.3 us here with whole histograms crossing the cluster and the scores loaded row by row, 54.8 with
// two-level histograms and every load in flight at once (score kernel 45 us of it).
//
// The kept set is the k items of largest (value, lowest index): as 64-bit keys
// (value bits, ~index) they are distinct, so the threshold is one key and an item is kept
// exactly when its key is not below it; no separate treatment of equal values.
#include <cooperative_groups.h>

#include <algorithm>

#include "bd_internal.h"
#include "bd_topk.cuh"

namespace cg = cooperative_groups;

namespace bd {

constexpr int kTMaxCluster = 8;     // CTAs per unit: the portable cluster size
constexpr int kTGroups = 64;        // groups of kTFine adjacent histogram bins
constexpr int kTFine = kBins / kTGroups;

struct TopkLongSmem {
  uint32_t bins[kBins];             // own histogram, then all ranks' boundary-bin items
  uint64_t cand[kBinCandMax];       // own boundary-bin items
  uint32_t digit[2][256];           // radix passes (crowded boundary bin)
  uint32_t wsum[32];
  float2 range[kTMaxCluster];       // every rank's (min, max)
  uint32_t group[kTMaxCluster][kTGroups];    // every rank's items per group of bins
  uint32_t fine[kTFine][kTMaxCluster];       // the boundary group's bins, every rank's
  uint32_t chosen[kTMaxCluster];    // every rank's kept positions
  uint32_t in_bin[kTMaxCluster];    // every rank's boundary-bin items
  float wmin[32], wmax[32];
  uint64_t key;
  uint32_t total, bin, above, count, n_cand, group_star, group_above;
  int first_kept;
};
static_assert(sizeof(uint32_t) * kBins >= sizeof(uint64_t) * kBinCandMax, "all ranks' items fit the bins");

// Inclusive scan over the 1024 threads (wsum scratch); *total gets the sum.
__device__ __forceinline__ uint32_t block_inclusive(uint32_t v, uint32_t* wsum, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, v, off);
    if (lane >= off) v += y;
  }
  if (lane == 31) wsum[warp] = v;
  __syncthreads();
  const uint32_t w = wsum[lane];
  const uint32_t below = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u);
  const uint32_t all = __reduce_add_sync(0xffffffffu, w);
  if (threadIdx.x == 0) *total = all;
  return v + below;
}

// ROWS: items per thread held in registers; 0: any number of items, re-read from the scores
// (L2) by each pass.  CHUNK: items are chunks of p.chunk positions, else positions.
template <int ROWS, bool CHUNK>
__global__ void __launch_bounds__(kTopkThreads, 1) topk_cluster_kernel(const TopkParams p, int C, int rows_per_cta) {
  __shared__ TopkLongSmem S;
  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)blockIdx.x % C, unit = (int)blockIdx.x / C;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");   // this CTA has started
  const float* sc = p.score + (size_t)unit * p.n_mid_pad;
  const int rows = rows_per_cta;                  // <= ROWS when ROWS > 0
  const int item0 = rank * rows * kTopkThreads;
  {   // the slice's scores on their way into L2 while the score kernel finishes
    const int s = CHUNK ? p.chunk : 1;
    const long long a = (long long)item0 * s, b = a + (long long)rows * kTopkThreads * s;
    if (a < p.n_mid_pad)
      prefetch_lines_l2(sc + a, (size_t)(min(b, (long long)p.n_mid_pad) - a) * 4, tid, kTopkThreads);
  }
  for (int i = tid; i < kBins; i += kTopkThreads) S.bins[i] = 0;
  if (tid == 0) S.n_cand = 0;
  grid_dependency_wait();
  allow_dependent_launch();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");             // every CTA is running

  const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 && rank == 0 ? p.status : nullptr);
  int32_t* out = p.idx_out + (size_t)unit * p.budget;
  const int gtid = rank * kTopkThreads + tid, gthreads = C * kTopkThreads;
  if (topk_keep_all(p, unit, t_u, out, gtid, gthreads)) return;
  const int lo = p.n_sink, hi = t_u - p.n_recent, n_pos = max(0, hi - lo);
  const int s = CHUNK ? p.chunk : 1;
  const int c_first = CHUNK ? lo / s : 0;
  const int n = CHUNK ? (n_pos > 0 ? (hi - 1) / s - c_first + 1 : 0) : n_pos;
  const int k = min((p.budget - p.n_sink - p.n_recent) / s, n);
  // members of item i: positions [a, b) (only the first and the last chunk can be short)
  auto members = [&](int i, int& a, int& b) {
    a = CHUNK ? max((c_first + i) * s, lo) : lo + i;
    b = CHUNK ? min((c_first + i + 1) * s, hi) : a + 1;
  };
  // fp32 bits of item i's score: non-negative, so their order is the values' (NaN counts as 0);
  // a chunk's members are summed in position order, eight loads in flight
  auto value = [&](int i) -> uint32_t {
    float v = 0.f;
    if (CHUNK) {
      int a, b;
      members(i, a, b);
      for (int q0 = a; q0 < b; q0 += 8) {
        float t[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) t[j] = q0 + j < b ? __ldcg(sc + (q0 + j - lo)) : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) v += t[j];
      }
    } else {
      v = __ldcg(sc + i);
    }
    return v > 0.f ? __float_as_uint(v) : 0u;
  };
  const int w_item0 = item0 + warp * rows * 32, w_end = min(n, w_item0 + 32 * rows);   // the warp's items
  constexpr uint32_t kNoItem = ~0u;               // past the items (a score's bits are never this)
  uint32_t u[ROWS > 0 ? ROWS : 1];
  if (ROWS > 0 && CHUNK) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int i = w_item0 + 32 * r + lane;
      u[r] = i < w_end ? value(i) : kNoItem;
    }
  } else if (ROWS > 0) {                          // all loads in flight before the first is used
    const float* base = sc + w_item0 + lane;
    const int left = w_end - w_item0 - lane;
    float x[ROWS > 0 ? ROWS : 1];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) x[r] = 32 * r < left ? __ldcg(base + 32 * r) : 0.f;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) u[r] = 32 * r < left ? (x[r] > 0.f ? __float_as_uint(x[r]) : 0u) : kNoItem;
  }
  // f(r, i, bits) for every item of this thread, in item order
  auto each = [&](auto f) {
    if constexpr (ROWS > 0) {
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        const int i = w_item0 + 32 * r + lane;
        if (u[r] != kNoItem) f(r, i, u[r]);
      }
    } else {
#pragma unroll 4
      for (int r = 0; r < rows; ++r) {
        const int i = w_item0 + 32 * r + lane;
        if (i < n) f(r, i, value(i));
      }
    }
  };
  auto key_of = [](int i, uint32_t bits) -> uint64_t {
    return (static_cast<uint64_t>(bits) << 32) | (0xFFFFFFFFu - (uint32_t)i);
  };

  uint64_t threshold = 0;                         // k == n: everything; k == 0: nothing (below)
  if (k > 0 && k < n) {
    // ---- value range of the unit
    float lmin = INFINITY, lmax = 0.f;
    each([&](int, int, uint32_t bits) {
      const float v = __uint_as_float(bits);
      lmin = fminf(lmin, v);
      lmax = fmaxf(lmax, v);
    });
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, off));
      lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
    }
    if (lane == 0) {
      S.wmin[warp] = lmin;
      S.wmax[warp] = lmax;
    }
    __syncthreads();
    if (warp == 0) {
      lmin = S.wmin[lane];
      lmax = S.wmax[lane];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        lmin = fminf(lmin, __shfl_xor_sync(0xffffffffu, lmin, off));
        lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, off));
      }
      if (lane < C) *cluster.map_shared_rank(&S.range[rank], lane) = make_float2(lmin, lmax);
    }
    cluster.sync();
    float vmin = INFINITY, vmax = 0.f;
    for (int q = 0; q < C; ++q) {
      vmin = fminf(vmin, S.range[q].x);
      vmax = fmaxf(vmax, S.range[q].y);
    }
    // ---- histogram, linear between min and max: the bin of the k-th largest item.  Any
    // scale >= 0 keeps the bins monotone in the value (an infinite range puts all in bin 0).
    const float scale = vmax > vmin ? (float)(kBins - 1) / (vmax - vmin) : 0.f;
    auto bin_of = [&](uint32_t bits) -> int {
      return min(kBins - 1, max(0, (int)((__uint_as_float(bits) - vmin) * scale)));
    };
    each([&](int, int, uint32_t bits) { atomicAdd(&S.bins[bin_of(bits)], 1u); });
    __syncthreads();
    // The boundary bin in two levels, so that little crosses the cluster: sums of 64 bins go to every
    // rank, then each reads the 64 bins of the group that holds the k-th item (every rank
    // reading every histogram whole, 1 MB per cluster, took 4.6 us against 1.5).
    static_assert(kBins == 4 * kTopkThreads && kTFine == 64 && kTGroups == 64, "16 threads sum a group of bins");
    {
      const uint4 h = reinterpret_cast<const uint4*>(S.bins)[tid];
      uint32_t sum = (h.x + h.y) + (h.z + h.w);
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
      if ((lane & 15) < C) *cluster.map_shared_rank(&S.group[rank][tid >> 4], lane & 15) = sum;
    }
    cluster.sync();
    // the entry of 64 (two per lane of warp 0) that holds the k-th item, `over` items being in
    // later entries than these 64: its index, items after it, its own
    auto find = [&](uint32_t h0, uint32_t h1, uint32_t in_all, uint32_t over, auto found) {
      uint32_t incl = h0 + h1;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += y;
      }
      const uint32_t after1 = over + in_all - incl, after0 = after1 + h1;
      if (after1 < (uint32_t)k && (uint32_t)k <= after1 + h1) found(2 * lane + 1, after1, h1);
      if (after0 < (uint32_t)k && (uint32_t)k <= after0 + h0) found(2 * lane, after0, h0);
    };
    if (warp == 0) {
      uint32_t h0 = 0, h1 = 0;
      for (int q = 0; q < C; ++q) {
        h0 += S.group[q][2 * lane];
        h1 += S.group[q][2 * lane + 1];
      }
      find(h0, h1, (uint32_t)n, 0u, [&](int g, uint32_t after, uint32_t own) {
        S.group_star = (uint32_t)g;
        S.group_above = after;
        S.total = own;
      });
    }
    __syncthreads();
    if (tid < kTFine * kTMaxCluster) {
      const int q = tid % kTMaxCluster, j = tid / kTMaxCluster;
      S.fine[j][q] = q < C ? cluster.map_shared_rank(S.bins, q)[S.group_star * kTFine + j] : 0u;
    }
    __syncthreads();
    if (warp == 0) {
      uint32_t h0 = 0, h1 = 0;
#pragma unroll
      for (int q = 0; q < kTMaxCluster; ++q) {
        h0 += S.fine[2 * lane][q];
        h1 += S.fine[2 * lane + 1][q];
      }
      find(h0, h1, S.total, S.group_above, [&](int j, uint32_t after, uint32_t own) {
        S.bin = S.group_star * kTFine + (uint32_t)j;
        S.above = after;
        S.count = own;
      });
    }
    __syncthreads();
    const int bstar = (int)S.bin;
    const uint32_t nc = S.count;
    if (nc <= (uint32_t)kBinCandMax) {
      // ---- the bin's items of every rank, ranked exactly
      if (tid < C) S.in_bin[tid] = S.fine[bstar % kTFine][tid];
      each([&](int, int i, uint32_t bits) {
        if (bin_of(bits) == bstar) S.cand[atomicAdd(&S.n_cand, 1u)] = key_of(i, bits);
      });
      cluster.sync();
      uint64_t* all = reinterpret_cast<uint64_t*>(S.bins);
      for (int i = tid; i < (int)nc; i += kTopkThreads) {
        int q = 0, j = i;
        while (j >= (int)S.in_bin[q]) j -= (int)S.in_bin[q++];
        all[i] = cluster.map_shared_rank(S.cand, q)[j];
      }
      __syncthreads();
      const uint32_t m = (uint32_t)k - S.above;   // rank (1-based) of the k-th item inside the bin
      for (int i = tid; i < (int)nc; i += kTopkThreads) {
        const uint64_t mine = all[i];
        uint32_t larger = 0;
        for (int j = 0; j < (int)nc; ++j) larger += all[j] > mine;
        if (larger == m - 1) S.key = mine;
      }
    } else {
      // ---- crowded bin (many equal or near-equal values): radix select on the keys, 8 bits
      // per pass; a pass's counts meet in every CTA, two buffers so that one barrier a pass
      // is enough
      uint64_t prefix = 0, mask = 0;
      uint32_t rem = (uint32_t)k;
      for (int pass = 0; pass < 8; ++pass) {
        const int shift = 56 - 8 * pass;
        uint32_t* d = S.digit[pass & 1];
        if (tid < 256) d[tid] = 0;
        __syncthreads();
        each([&](int, int i, uint32_t bits) {
          const uint64_t key = key_of(i, bits);
          if ((key & mask) == prefix) atomicAdd(&d[(uint32_t)(key >> shift) & 255u], 1u);
        });
        cluster.sync();
        uint32_t h = 0;
        if (tid < 256)
          for (int q = 0; q < C; ++q) h += cluster.map_shared_rank(d, q)[tid];
        const uint32_t upto = block_inclusive(h, S.wsum, &S.total);
        __syncthreads();
        const uint32_t over = S.total - upto;     // matching items of a higher digit
        if (tid < 256 && over < rem && rem <= over + h) {
          S.key = prefix | (static_cast<uint64_t>(tid) << shift);
          S.above = over;
        }
        __syncthreads();
        prefix = S.key;
        rem -= S.above;
        mask |= static_cast<uint64_t>(0xFF) << shift;
        __syncthreads();
      }
    }
    __syncthreads();
    threshold = S.key;
  }

  // ---- kept positions of every rank, then the writes in position order
  const bool any = k > 0;
  uint32_t masks[ROWS > 0 ? ROWS : 1];
  uint32_t cnt = 0;                               // the warp's kept items
  if constexpr (ROWS > 0) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int i = w_item0 + 32 * r + lane;
      masks[r] = __ballot_sync(0xffffffffu, any && u[r] != kNoItem && key_of(i, u[r]) >= threshold);
      cnt += __popc(masks[r]);
    }
  } else {
    for (int r = 0; r < rows; ++r) {
      const int i = w_item0 + 32 * r + lane;
      cnt += __popc(__ballot_sync(0xffffffffu, any && i < n && key_of(i, value(i)) >= threshold));
    }
  }
  // an item takes s positions, the first and the last chunk perhaps fewer
  int short0 = 0, short1 = 0;
  if (CHUNK && n > 0) {
    int a, b;
    members(0, a, b);
    short0 = s - (b - a);
    members(n - 1, a, b);
    short1 = n > 1 ? s - (b - a) : 0;
  }
  if (tid == 0) S.first_kept = CHUNK && rank == 0 && any && n > 0 && key_of(0, value(0)) >= threshold ? 1 : 0;
  bool last_kept = false;
  if (CHUNK && short1 > 0 && n - 1 >= item0 && n - 1 < item0 + rows * kTopkThreads)
    last_kept = any && key_of(n - 1, value(n - 1)) >= threshold;
  const uint32_t incl = block_inclusive(lane == 31 ? cnt : 0u, S.wsum, &S.total);
  const uint32_t warp_base = __shfl_sync(0xffffffffu, incl, 31) - cnt;   // kept items of the warps before
  __syncthreads();
  const int cut = S.first_kept ? short0 : 0;
  const uint32_t my_chosen = S.total * (uint32_t)s - (uint32_t)cut - (last_kept ? (uint32_t)short1 : 0u);
  if (tid < C) *cluster.map_shared_rank(&S.chosen[rank], tid) = my_chosen;
  cluster.sync();                                 // no remote access after this
  int base = lo, chosen = 0;
  for (int q = 0; q < C; ++q) {
    base += q < rank ? (int)S.chosen[q] : 0;
    chosen += (int)S.chosen[q];
  }
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t run = warp_base;
  auto write = [&](int i, uint32_t order) {       // item i is the order-th kept one of this CTA
    int o = base + (int)order * s - (i > 0 ? cut : 0);
    int a, b;
    members(i, a, b);
    for (int q = a; q < b; ++q, ++o)
      if (o < p.budget) out[o] = q;
  };
  if constexpr (ROWS > 0) {
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const uint32_t mk = masks[r];
      if (mk == 0u) continue;                     // warp-uniform: most rows hold no kept item
      if ((mk >> lane) & 1u) write(w_item0 + 32 * r + lane, run + __popc(mk & lt));
      run += __popc(mk);
    }
  } else {
    for (int r = 0; r < rows; ++r) {
      const int i = w_item0 + 32 * r + lane;
      const uint32_t mk = __ballot_sync(0xffffffffu, any && i < n && key_of(i, value(i)) >= threshold);
      if ((mk >> lane) & 1u) write(i, run + __popc(mk & lt));
      run += __popc(mk);
    }
  }
  const int count = lo + chosen + p.n_recent;
  for (int i = gtid; i < lo; i += gthreads) out[i] = i;
  for (int i = gtid; i < p.n_recent; i += gthreads) out[lo + chosen + i] = hi + i;
  for (int i = count + gtid; i < p.budget; i += gthreads) out[i] = -1;
  if (gtid == 0) p.count_out[unit] = count;
}

// Selections that rank nothing: everything is kept, or the sinks and the recent window only.
__global__ void __launch_bounds__(256) topk_plain_kernel(const TopkParams p) {
  grid_dependency_wait();
  allow_dependent_launch();
  const int tid = threadIdx.x, unit = blockIdx.x;
  const int t_u = unit_context(p.seq_lens, unit, p.h_kv, p.t_ctx, tid == 0 ? p.status : nullptr);
  int32_t* out = p.idx_out + (size_t)unit * p.budget;
  if (topk_keep_all(p, unit, t_u, out, tid, 256)) return;
  const int lo = p.n_sink, hi = t_u - p.n_recent, count = lo + p.n_recent;
  for (int i = tid; i < p.budget; i += 256) out[i] = i < lo ? i : (i < count ? hi + (i - lo) : -1);
  if (tid == 0) p.count_out[unit] = count;
}

// ============================================================================ host side

cudaError_t launch_topk_plain(const TopkParams& p, int units, cudaStream_t stream) {
  TopkParams q = p;
  void* args[] = {&q};
  return launch_kernel(reinterpret_cast<void*>(&topk_plain_kernel), dim3(units), dim3(256), 0, stream, args, 0);
}

cudaError_t launch_topk_long(const TopkParams& p, int units, int n_items, cudaStream_t stream) {
  // CTAs per unit: enough to hold the items in registers, and more while a thread has over
  // eight positions to read and the GPU has SMs for all the CTAs.  A select call of 8 units:
  // 32K positions 30.2 / 26.5 / 28.0 us with 2 / 4 / 8 CTAs, 128K positions 107.7 / 83.3 /
  // 70.2 us; of 24 units of 36K positions 64.5 / 55.4 us with 2 / 4, and 70.1 us with 8 (192
  // CTAs, two waves).
  const bool chunked = p.chunk > 1;
  const int max_rows = chunked ? 8 : 16;
  const long n_pos = (long)n_items * p.chunk;
  int C = 2;
  while (C < kTMaxCluster && ((long)C * max_rows * kTopkThreads < n_items ||
                              (n_pos > (long)C * 8 * kTopkThreads && (long)2 * C * units <= current_sm_count())))
    C *= 2;
  int rows = std::max(1, (n_items + C * kTopkThreads - 1) / (C * kTopkThreads));
  TopkParams q = p;
  void* args[] = {&q, &C, &rows};
  void* fn = nullptr;
#define BD_TK(R)                                                                                  \
  if (!fn && rows <= R && R <= max_rows)                                                            \
    fn = chunked ? reinterpret_cast<void*>(&topk_cluster_kernel<(R < 16 ? R : 0), true>)            \
                 : reinterpret_cast<void*>(&topk_cluster_kernel<R, false>);
  BD_TK(1) BD_TK(2) BD_TK(4) BD_TK(8) BD_TK(16)
#undef BD_TK
  if (!fn)
    fn = chunked ? reinterpret_cast<void*>(&topk_cluster_kernel<0, true>)
                 : reinterpret_cast<void*>(&topk_cluster_kernel<0, false>);
  return launch_kernel(fn, dim3((unsigned)(C * units)), dim3(kTopkThreads), 0, stream, args, C);
}

}  // namespace bd
