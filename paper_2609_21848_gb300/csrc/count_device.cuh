// Device building blocks shared by the single-graph kernels (count.cu) and
// the batched kernels (batch.cu): packed wedge counters, the incremental
// Lemma 1 contribution, shared-memory hashing, the warp walk over a pivot's
// lower neighbours, and one window of the hub sweep.
#pragma once

#include <type_traits>

#include "internal.h"
#include "common.cuh"

namespace dbbc {

// Hash counters of the light and medium tiers: one 32-bit word per endpoint,
// (asym << 16) | sym. A count never exceeds the pivot's accepted wedges, and
// those are at most kMediumMaxWork in these tiers. One 32-bit shared atomic
// adds a wedge; a 64-bit shared add would be a compare-and-swap loop.
static_assert(kMediumMaxWork < 65536, "hash counters have 16-bit halves");

__device__ __forceinline__ uint32_t hash_slot(uint32_t w, int log_h) {
  return (w * 2654435769u) >> (32 - log_h);
}

// Find or insert endpoint w in a shared table of 2^log_h slots and add inc;
// returns the counter's previous value through *old. Returns false if the
// probe sequence ran past the table (cannot happen when the table has more
// slots than the pivot's accepted wedges).
__device__ __forceinline__ bool smem_hash_add(uint32_t* keys, uint32_t* vals, int log_h, uint32_t w, uint32_t inc,
                                              uint32_t* old) {
  const uint32_t mask = (1u << log_h) - 1u;
  uint32_t h = hash_slot(w, log_h);
  for (uint32_t probe = 0; probe <= mask; probe++) {
    uint32_t cur = *reinterpret_cast<volatile uint32_t*>(&keys[h]);
    if (cur == kEmptyKey) cur = atomicCAS(&keys[h], kEmptyKey, w);
    if (cur == kEmptyKey || cur == w) {
      *old = atomicAdd(&vals[h], inc);
      return true;
    }
    h = (h + 1u) & mask;
  }
  return false;
}

// Empty the first 2^log_h slots (log_h >= 5, both arrays 16-byte aligned) with
// `threads` threads, thread `t` of them.
__device__ __forceinline__ void hash_clear(uint32_t* keys, uint32_t* vals, int log_h, int t, int threads) {
  uint4* k4 = reinterpret_cast<uint4*>(keys);
  uint4* v4 = reinterpret_cast<uint4*>(vals);
  for (int i = t; i < (1 << log_h) / 4; i += threads) {
    k4[i] = make_uint4(kEmptyKey, kEmptyKey, kEmptyKey, kEmptyKey);
    v4[i] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// Smallest 2^k >= (work << mult_log) slots (at least 32, at most 2^max_log).
// The tiers keep work <= 2^(max_log - 1), so a table always has more slots
// than the pivot has accepted wedges (and hence distinct endpoints).
__device__ __forceinline__ int table_log(uint64_t work, int max_log, int mult_log) {
  int k = 5;
  while (k < max_log && (1ull << k) < (work << mult_log)) k++;
  return k;
}

struct PivotGeom {
  int64_t rb;    // row start of the pivot
  uint32_t L;    // lower neighbours
  uint32_t lim;  // entries x < lim are accepted endpoints: (side_rank(p) << 1)
  int64_t base;  // first row of the other side
};

__device__ __forceinline__ PivotGeom pivot_geom(const CsrView& g, int32_t p) {
  PivotGeom q;
  const bool ok = DBBC_CHECK(p >= 0 && p < g.n);  // checked builds: a bad pivot walks no neighbour
  if (!ok) p = 0;
  q.rb = g.row_ptr[p];
  q.L = ok ? g.lower[p] : 0u;
#if DBBC_CHECKED
  if (q.L && !DBBC_CHECK(q.rb >= 0 && q.rb + q.L <= g.row_ptr[p + 1] && g.row_ptr[p + 1] <= g.nnz)) q.L = 0;
#endif
  const bool is_u = p < g.n_u;
  q.lim = (is_u ? (uint32_t)p : (uint32_t)(p - g.n_u)) << 1;
  q.base = is_u ? (int64_t)g.n_u : 0;
  return q;
}

// Span [b, en) of the row of the vertex of the other side named by the CSR
// entry e of a pivot with geometry q. Checked builds test the row index and
// bounds; a failed test gives an empty span.
__device__ __forceinline__ void neighbour_row(const CsrView& g, const PivotGeom& q, uint32_t e, uint32_t& b,
                                              uint32_t& en) {
  const int64_t vrow = q.base + (e >> 1);
  b = en = 0;
  if (DBBC_CHECK(vrow >= 0 && vrow < g.n)) {
    const uint2 s = g.span[vrow];
    if (DBBC_CHECK((int64_t)s.x >= g.row_ptr[vrow] && s.x <= s.y && (int64_t)s.y <= g.row_ptr[vrow + 1])) {
      b = s.x;
      en = s.y;
    }
  }
}

// Hash tiers: groups of G lanes (group gid of `groups`) take lower neighbours
// gid, gid + groups, ... of the pivot; a group walks its neighbour's accepted
// prefix G entries at a time. visit(G, x, e, i, pos, last) is called by the
// whole warp for every chunk: the lane's entry x at CSR position pos (~0 where
// nothing is accepted) of the row of neighbour position i, whose entry in the
// pivot's row is e; `last` says that the neighbour ends with this chunk (so it
// is called with `last` exactly once per neighbour).
// The walk is bound by the latency of its dependent loads (entry of the
// pivot's row, row bounds, entries), so each is issued ahead: the next chunk
// (of this neighbour, or the first of the group's next one) before the current
// one is visited, row bounds one neighbour ahead and row entries two. Every
// group moves on to its next neighbour by itself. The loop's only exit is a vote
// of the whole warp, so its trip count is warp-uniform and every lane reaches
// every vote and shuffle in it; a group that has run out only votes. Lanes
// diverge inside visit alone, and meet again at the __syncwarp after it. With 32-bit
// counters (kHashSlotBytes, which also lets half again as many CTAs fit an SM)
// this took the 20M-edge rating graph's medium tier from 0.99 to 0.44 ms and a
// 1M-edge one's from 92 to 47 us (light: 80 to 52 us), 1,024 batched small
// graphs' light tier from 0.90 to 0.54 ms.
template <int G, typename Visit>
__device__ __forceinline__ void group_walk(uint32_t gid, uint32_t groups, const CsrView& g, const PivotGeom& q,
                                           Visit&& visit) {
  const unsigned lane = lane_id();
  const uint32_t gl = lane & (G - 1);
  const uint32_t* __restrict__ col = g.col;
  auto bounds = [&](bool ok, uint32_t e, uint32_t& c, uint32_t& en) {
    c = en = 0;
    if (ok) neighbour_row(g, q, e, c, en);
  };
  uint32_t i = gid;
  uint32_t e = i < q.L ? col[q.rb + i] : 0u;
  uint32_t e1 = i + groups < q.L ? col[q.rb + i + groups] : 0u;
  uint32_t c, en, c1, en1;
  bounds(i < q.L, e, c, en);
  uint32_t x = en - c > gl ? col[c + gl] : 0xFFFFFFFFu;
  bounds(i + groups < q.L, e1, c1, en1);
  uint32_t e2 = i + 2 * groups < q.L ? col[q.rb + i + 2 * groups] : 0u;
  while (__any_sync(kFullMask, i < q.L)) {
    const bool cont = __shfl_sync(kFullMask, x, lane | (G - 1)) < q.lim;  // all accepted: the row goes on
    const uint32_t xc = x < q.lim ? x : 0xFFFFFFFFu, ec = e, ic = i, pos = c + gl;
    if (cont) {
      c += G;
    } else {
      i += groups;
      c = c1;
      en = en1;
      e = e1;
    }
    x = en - c > gl ? col[c + gl] : 0xFFFFFFFFu;
    if (!cont) {
      e1 = e2;
      bounds(i + groups < q.L, e1, c1, en1);
      e2 = i + 2 * groups < q.L ? col[q.rb + i + 2 * groups] : 0u;
    }
    visit(std::integral_constant<int, G>(), xc, ec, ic, pos, !cont && ic < q.L);
    __syncwarp();
  }
}

template <typename Visit>
__device__ __forceinline__ void group_walk_dispatch(int group_log, uint32_t tid, uint32_t threads, const CsrView& g,
                                                    const PivotGeom& q, Visit&& visit) {
  switch (group_log) {
    case 2: group_walk<4>(tid >> 2, threads >> 2, g, q, visit); break;
    case 3: group_walk<8>(tid >> 3, threads >> 3, g, q, visit); break;
    case 4: group_walk<16>(tid >> 4, threads >> 4, g, q, visit); break;
    default: group_walk<32>(tid >> 5, threads >> 5, g, q, visit); break;
  }
}

// Count a pivot's wedges into a hash table and add their Lemma 1
// contributions. A pivot's sums fit 32 bits (at most kMediumMaxWork wedges,
// each adding less than that). Returns false if the table ran out of slots.
__device__ __forceinline__ bool hash_count(int group_log, uint32_t tid, uint32_t threads, const CsrView& g,
                                           const PivotGeom& q, uint32_t* keys, uint32_t* vals, int log_h,
                                           uint64_t& bal, uint64_t& unb) {
  bool fits = true;
  uint32_t own = 0, other = 0;
  group_walk_dispatch(group_log, tid, threads, g, q, [&](auto, uint32_t x, uint32_t e, uint32_t, uint32_t, bool) {
    if (x != 0xFFFFFFFFu) {
      const uint32_t sh = ((x ^ e) & 1u) << 4;
      uint32_t old = 0;
      fits &= smem_hash_add(keys, vals, log_h, x >> 1, 1u << sh, &old);
      const uint32_t v = __funnelshift_l(old, old, sh);  // (other class << 16) | own class
      own += v & 0xFFFFu;
      other += v >> 16;
    }
  });
  bal += own;
  unb += other;
  return fits;
}

// log2 of the lanes per neighbour for a pivot whose lower neighbours carry
// `work` accepted wedges in all (at least 4 lanes, at most `max_log`).
__device__ __forceinline__ int hash_group_log(uint64_t work, uint32_t L, int max_log) {
  const uint64_t mean = work / (L ? L : 1);
  const int lg = mean >= 24 ? 5 : mean >= 12 ? 4 : mean >= 6 ? 3 : 2;
  return lg < max_log ? lg : max_log;
}

// log2 of the hash slots a tier's tables need at most: table_log of the
// tier's largest accepted-wedge count (5..cap). Kernels of a tier get this
// many slots per table, so small tiers leave room for more CTAs per SM.
inline int tier_slots_log(uint64_t max_work, int mult_log, int cap) {
  int k = 5;
  while (k < cap && (1ull << k) < (max_work << mult_log)) k++;
  return k;
}

constexpr int kLightWarps = 8;
constexpr size_t kHashSlotBytes = 8;  // a key and a packed counter

constexpr int kMediumThreads = 256;
constexpr int kMediumWarps = kMediumThreads / 32;

// ------------------------------------------------------------------ hub tier
// Window sweep. A hub pivot's accepted endpoints [0, side_rank(p)) are cut
// into windows of kSweepWindow16 (or kSweepWindow32) consecutive side ranks. A
// work item is one hub and a span of its windows, owned by one CTA, so the
// counts of every endpoint in a window are complete inside that CTA: they live
// in shared memory, and the Lemma 1 contributions come from the value each
// atomic returns. Each lower neighbour v keeps a cursor into its row (uint32
// positions: a CSR has fewer than 2^32 entries); rows ascend, so sweeping the
// windows in order moves every cursor forward only. Counters pack
// (asym << 16) | sym when the hub has fewer than 2^16 lower neighbours (no
// count can exceed that), else (asym << 32) | sym.
constexpr int kSweepThreads = DBBC_SWEEP_THREADS;
static_assert(kSweepWindow16 % 4 == 0, "window buffers are cleared 16 bytes at a time");

// Clear the first `words` 32-bit words of a window (16 bytes per store; the
// window buffer holds a multiple of 4 words).
template <int THREADS = kSweepThreads>
__device__ __forceinline__ void zero_words(uint32_t* w, uint32_t words) {
  uint4* q = reinterpret_cast<uint4*>(w);
  const uint32_t quads = (words + 3) >> 2;
  for (uint32_t j = threadIdx.x; j < quads; j += THREADS) q[j] = make_uint4(0u, 0u, 0u, 0u);
}

// Counter widths of a window. CW = 16: one 32-bit word per endpoint packing
// (asym << 16) | sym, kSweepWindow16 ranks per window. CW = 8: two endpoints
// per 32-bit word, each (asym << 8) | sym, twice the ranks per window; used
// where every endpoint has degree < 256 or the hub has fewer than 256 lower
// neighbours (a count never exceeds either). CW = 4: four endpoints per word,
// each (asym << 4) | sym, four times the ranks, where counts stay below 16.
// CW = 32: one 64-bit word per endpoint, half the ranks.
// W16: the window's 16-bit counters (kSweepWindow16, or kHalfWindow16 in the half
// CTAs of small graphs).
template <int CW, uint32_t W16 = kSweepWindow16>
__host__ __device__ constexpr uint32_t window_ranks() {
  return CW == 4 ? 4 * W16 : CW == 8 ? 2 * W16 : CW == 16 ? W16 : W16 / 2;
}

// The windows of a work item: quarter ones over [lo, qe), tiny ones over
// [qe, te), narrow ones over [te, ne), wide ones over [ne, hi), numbered in
// rank order.
template <uint32_t W16>
struct ItemWindowsOf {
  uint32_t lo, qe, te, ne, hi;
  uint32_t rq, rt, rn, rw;
  ItemWindowsOf() = default;
  __device__ __forceinline__ explicit ItemWindowsOf(const SweepItem& it) {
    lo = it.lo;
    hi = it.hi;
    qe = min(max(it.q_end, lo), hi);
    te = min(max(it.t_end, qe), hi);
    ne = min(max(it.n_end, te), hi);
    rq = (qe - lo + window_ranks<4, W16>() - 1) / window_ranks<4, W16>();
    rt = (te - qe + window_ranks<8, W16>() - 1) / window_ranks<8, W16>();
    rn = (ne - te + window_ranks<16, W16>() - 1) / window_ranks<16, W16>();
    rw = (hi - ne + window_ranks<32, W16>() - 1) / window_ranks<32, W16>();
  }
  __device__ __forceinline__ uint32_t count() const { return rq + rt + rn + rw; }
  // window r: its ranks [wlo, whi) and counter width
  __device__ __forceinline__ void window(uint32_t r, uint32_t& wlo, uint32_t& whi, int& cw) const {
    if (r < rq) {
      wlo = lo + r * window_ranks<4, W16>();
      whi = min(wlo + window_ranks<4, W16>(), qe);
      cw = 4;
    } else if (r < rq + rt) {
      wlo = qe + (r - rq) * window_ranks<8, W16>();
      whi = min(wlo + window_ranks<8, W16>(), te);
      cw = 8;
    } else if (r < rq + rt + rn) {
      wlo = te + (r - rq - rt) * window_ranks<16, W16>();
      whi = min(wlo + window_ranks<16, W16>(), ne);
      cw = 16;
    } else {
      wlo = ne + (r - rq - rt - rn) * window_ranks<32, W16>();
      whi = min(wlo + window_ranks<32, W16>(), hi);
      cw = 32;
    }
  }
  // the window holding rank x (lo <= x < hi)
  __device__ __forceinline__ uint32_t index_of(uint32_t x) const {
    if (x < qe) return (x - lo) / window_ranks<4, W16>();
    if (x < te) return rq + (x - qe) / window_ranks<8, W16>();
    if (x < ne) return rq + rt + (x - te) / window_ranks<16, W16>();
    return rq + rt + rn + (x - ne) / window_ranks<32, W16>();
  }
};
using ItemWindows = ItemWindowsOf<kSweepWindow16>;

}  // namespace dbbc
