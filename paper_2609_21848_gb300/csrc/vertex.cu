// Butterflies containing each vertex (the "tip" input of the paper's
// applications) and each edge (the "wing" input), computed with the same
// tiers as the totals. Once the buckets of a pivot u are complete (a pivot's
// hash table, or one window of a hub):
//   * every endpoint w and u itself are in C(p,2) + C(q,2) balanced and p*q
//     unbalanced butterflies of u, where (p, q) are w's symmetric and
//     asymmetric bucket counts (Algorithm 1, Lemma 1);
//   * a symmetric wedge u-v-w pairs with the p - 1 other symmetric wedges to w
//     (balanced) and the q asymmetric ones (unbalanced); an asymmetric wedge
//     with q - 1 and p. Each pairing is one butterfly through the middle v and
//     through both edges (u, v) and (v, w) of the wedge.
// The middles and edges need a second walk of the same wedges after the counts
// are final. Vertex results are accumulated per CSR row and mapped to unified
// ids at the end; edge results per CSR position (an edge has one position in
// each of its two rows), summed over both positions when an edge is queried.
#include "sweep_device.cuh"

namespace dbbc {

struct TipOut {
  unsigned long long* vb = nullptr;  // [n] per row (vertex counts)
  unsigned long long* vu = nullptr;
  unsigned long long* eb = nullptr;  // [nnz] per CSR position (edge counts); when no edge can be in 2^32
  unsigned long long* eu = nullptr;  // butterflies, eu is null and eb holds (unbalanced << 32) | balanced
  int64_t n = 0, nnz = 0;            // their lengths
};

// Counter of endpoint w in a shared hash table (the key must be present).
__device__ __forceinline__ uint32_t hash_find(const uint32_t* keys, const uint32_t* vals, int log_h, uint32_t w) {
  const uint32_t mask = (1u << log_h) - 1u;
  uint32_t h = hash_slot(w, log_h);
  for (uint32_t probe = 0; probe <= mask; probe++) {
    if (keys[h] == w) return vals[h];
    if (keys[h] == kEmptyKey) break;
    h = (h + 1u) & mask;
  }
  return 0u;
}

// Butterflies one wedge is in, from its endpoint's buckets (p, q) packed as
// (q << 32) | p: the other wedges of its own class close balanced ones, the
// wedges of the other class unbalanced ones.
__device__ __forceinline__ void wedge_pairs(unsigned long long packed, bool sym, uint64_t& bal, uint64_t& unb) {
  const uint64_t p = packed & 0xFFFFFFFFull, q = packed >> 32;
  bal = sym ? p - 1 : q - 1;
  unb = sym ? q : p;
}

__device__ __forceinline__ void endpoint_contrib(unsigned long long packed, uint64_t& bal, uint64_t& unb) {
  const uint64_t p = packed & 0xFFFFFFFFull, q = packed >> 32;
  bal += (p * (p - (p > 0)) >> 1) + (q * (q - (q > 0)) >> 1);
  unb += p * q;
}

__device__ __forceinline__ void add_pair(unsigned long long* b, unsigned long long* u, int64_t i, uint64_t x,
                                         uint64_t y) {
  if (x) atomicAdd(&b[i], (unsigned long long)x);
  if (y) atomicAdd(&u[i], (unsigned long long)y);
}

// Per-row (vertex) and per-CSR-position (edge) sums; checked builds test the
// position first.
__device__ __forceinline__ void add_vertex(const TipOut& o, int64_t r, uint64_t x, uint64_t y) {
  if (DBBC_CHECK(r >= 0 && r < o.n)) add_pair(o.vb, o.vu, r, x, y);
}
__device__ __forceinline__ void add_edge(const TipOut& o, int64_t j, uint64_t x, uint64_t y) {
  if (!DBBC_CHECK(j >= 0 && j < o.nnz)) return;
  if (o.eu) add_pair(o.eb, o.eu, j, x, y);
  else if (x | y) atomicAdd(&o.eb[j], (unsigned long long)(x | (y << 32)));
}

// The endpoints of a pivot's complete hash table (slots t, t + threads, ...):
// each endpoint and the pivot get the endpoint's Lemma 1 totals; the pivot's
// share is summed over the warp.
__device__ __forceinline__ void credit_endpoints(const CsrView& g, int32_t p, const uint32_t* keys,
                                                 const uint32_t* vals, int log_h, int t, int threads,
                                                 const TipOut& o) {
  const int64_t end_base = p < g.n_u ? 0 : (int64_t)g.n_u;  // endpoints share the pivot's side
  uint64_t pb = 0, pu = 0;
  for (int i = t; i < (1 << log_h); i += threads) {
    const uint32_t v = vals[i];
    if (v) {
      uint64_t eb = 0, eu = 0;
      endpoint_contrib(((unsigned long long)(v >> 16) << 32) | (v & 0xFFFFu), eb, eu);
      add_vertex(o, end_base + keys[i], eb, eu);
      pb += eb;
      pu += eu;
    }
  }
  pb = warp_sum_u64(pb);
  pu = warp_sum_u64(pu);
  if (lane_id() == 0) add_vertex(o, p, pb, pu);
}

// The second walk over a light or medium pivot's wedges, by the same lane
// groups as the first: each lane credits the far edge (v, w) of its wedge from
// the endpoint's final counter; when a group reaches the end of a neighbour v
// its lanes' sums credit the middle v and the near edge (u, v). Sums fit 32
// bits (at most kMediumMaxWork wedges of fewer butterflies each). Lane groups
// sized to the pivot's mean segment keep the warp's lanes busy where one warp
// per neighbour left most of them idle (mean accepted segments are 5 to 20
// entries in these tiers): per-edge counts of a 20M-edge graph, medium tier
// 4.06 to 0.74 ms and light 1.41 to 0.40 ms; per-vertex counts of a 4M-edge
// one, 1.21 to 0.26 ms and 0.42 to 0.14 ms.
template <bool VERT, bool EDGE>
__device__ __forceinline__ void second_walk(int group_log, uint32_t tid, uint32_t threads, const CsrView& g,
                                            const PivotGeom& q, const uint32_t* keys, const uint32_t* vals, int log_h,
                                            const TipOut& o) {
  uint32_t sb = 0, su = 0;
  group_walk_dispatch(group_log, tid, threads, g, q,
                      [&](auto gtag, uint32_t x, uint32_t e, uint32_t i, uint32_t pos, bool last) {
    constexpr int G = decltype(gtag)::value;
    if (x != 0xFFFFFFFFu) {
      const uint32_t v = hash_find(keys, vals, log_h, x >> 1);
      uint64_t cb, cu;
      wedge_pairs(((unsigned long long)(v >> 16) << 32) | (v & 0xFFFFu), ((x ^ e) & 1u) == 0, cb, cu);
      if (EDGE) add_edge(o, pos, cb, cu);
      sb += (uint32_t)cb;
      su += (uint32_t)cu;
    }
    __syncwarp();
    if (__any_sync(kFullMask, last)) {
      uint32_t tb = sb, tu = su;
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) {
        tb += __shfl_xor_sync(kFullMask, tb, off);
        tu += __shfl_xor_sync(kFullMask, tu, off);
      }
      if (last) {
        if ((threadIdx.x & (G - 1)) == 0) {
          if (VERT) add_vertex(o, q.base + (e >> 1), tb, tu);
          if (EDGE) add_edge(o, q.rb + i, tb, tu);
        }
        sb = su = 0;
      }
    }
  });
}

// ------------------------------------------------------------------ light / medium
// Tables as in the counting kernels (2^slots_log slots).
template <bool VERT, bool EDGE>
__global__ void __launch_bounds__(kLightWarps * 32) tips_light_kernel(CsrView g, const int32_t* __restrict__ piv,
                                                                      const uint64_t* __restrict__ work,
                                                                      int64_t n_piv, int hash_mult_log, int slots_log,
                                                                      TipOut o, unsigned* status) {
  extern __shared__ __align__(16) unsigned char light_smem[];
  const int slots = 1 << slots_log;
  const int w = threadIdx.x >> 5;
  const unsigned lane = lane_id();
  uint32_t* keys = reinterpret_cast<uint32_t*>(light_smem) + 2 * w * slots;
  uint32_t* vals = keys + slots;
  hash_clear(keys, vals, slots_log, lane, 32);
  __syncwarp();
  bool full = false;
  const int64_t nw = (int64_t)gridDim.x * kLightWarps;
  for (int64_t t = (int64_t)blockIdx.x * kLightWarps + w; t < n_piv; t += nw) {
    const int32_t p = piv[t];
    const uint64_t wp = work[p];
    const int log_h = table_log(wp, slots_log, hash_mult_log);
    const PivotGeom q = pivot_geom(g, p);
    const int gl = hash_group_log(wp, q.L, 5);
    uint64_t unused_b = 0, unused_u = 0;
    full |= !hash_count(gl, lane, 32u, g, q, keys, vals, log_h, unused_b, unused_u);
    if (VERT) credit_endpoints(g, p, keys, vals, log_h, lane, 32, o);
    second_walk<VERT, EDGE>(gl, lane, 32u, g, q, keys, vals, log_h, o);
    hash_clear(keys, vals, log_h, lane, 32);
    __syncwarp();
  }
  if (full) atomicOr(status, DBBC_DEV_HASH_FULL);
}

template <bool VERT, bool EDGE>
__global__ void __launch_bounds__(kMediumThreads) tips_medium_kernel(CsrView g, const int32_t* __restrict__ piv,
                                                                     const uint64_t* __restrict__ work,
                                                                     int64_t n_piv, int hash_mult_log, int slots_log,
                                                                     TipOut o, unsigned* status) {
  extern __shared__ __align__(16) unsigned char med_smem[];
  uint32_t* keys = reinterpret_cast<uint32_t*>(med_smem);
  uint32_t* vals = keys + (1 << slots_log);
  hash_clear(keys, vals, slots_log, threadIdx.x, kMediumThreads);
  __syncthreads();
  bool full = false;
  for (int64_t t = blockIdx.x; t < n_piv; t += gridDim.x) {
    const int32_t p = piv[t];
    const uint64_t wp = work[p];
    const int log_h = table_log(wp, slots_log, hash_mult_log);
    const PivotGeom q = pivot_geom(g, p);
    const int gl = hash_group_log(wp, q.L, 5);
    uint64_t unused_b = 0, unused_u = 0;
    full |= !hash_count(gl, threadIdx.x, (uint32_t)kMediumThreads, g, q, keys, vals, log_h, unused_b, unused_u);
    __syncthreads();
    if (VERT) credit_endpoints(g, p, keys, vals, log_h, threadIdx.x, kMediumThreads, o);
    second_walk<VERT, EDGE>(gl, threadIdx.x, (uint32_t)kMediumThreads, g, q, keys, vals, log_h, o);
    __syncthreads();
    hash_clear(keys, vals, log_h, threadIdx.x, kMediumThreads);
    __syncthreads();
  }
  if (full) atomicOr(status, DBBC_DEV_HASH_FULL);
}

// ------------------------------------------------------------------ hub windows
// A hub window runs in three passes over shared-memory counters: the window is
// counted (the counting sweep's walk without returned values), its endpoints
// are credited, and the segments just counted are walked again for the middles
// and the edges. The first pass lists the segments it finds, so the last one
// visits only neighbours with entries in the window. Per-edge counts of the
// 20M-edge rating graph: sweep 31.4 -> 19.8 ms (half of it from both counts of
// an edge sharing one word, see dbbc_count_edges); it is bound by the latency
// of its loads and of the far edges' adds, 1.2e9 sectors to L2. Per-vertex
// counts of a 4M-edge one: 3.34 -> 2.26 ms, bound by issue slots (63%).

// A neighbour's segment [c, end) inside the current window; e: its entry in
// the hub's row, i: its position there.
struct Segment {
  uint32_t c, end, e, i;
};

// Shared byte address of the counter word of entry x's endpoint (see Win).
template <int CW>
__device__ __forceinline__ uint32_t counter_addr(uint32_t x, uint32_t wb) {
  return CW == 4 ? wb + ((x >> 1) & ~3u) : CW == 8 ? wb + (x & ~3u) : CW == 16 ? wb + ((x >> 1) << 2)
                                                                               : wb + ((x >> 1) << 3);
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

// Final counts of entry x's endpoint: of the wedge's own class and of the
// other one.
template <int CW>
__device__ __forceinline__ void counter_pair(uint32_t x, uint32_t s1, const Win& w, uint32_t& own, uint32_t& other) {
  const uint32_t addr = counter_addr<CW>(x, w.wb);
  own = 1u;  // checked builds: an address outside the window credits nothing
  other = 0u;
#if DBBC_CHECKED
  if (!DBBC_CHECK(x >= w.l && x < w.h && addr >= w.s_lo && addr + (CW == 32 ? 8u : 4u) <= w.s_hi)) return;
#endif
  if constexpr (CW == 32) {
    const uint32_t asym = ((x ^ s1) & 1u) << 2;
    own = lds_u32(addr + asym);
    other = lds_u32(addr + (asym ^ 4u));
  } else {
    const uint32_t v = lds_u32(addr);
    if constexpr (CW == 4) {
      const uint32_t sel = (x ^ s1) & 7u;
      own = (v >> (sel << 2)) & 0xFu;
      other = (v >> ((sel ^ 1u) << 2)) & 0xFu;
    } else if constexpr (CW == 8) {
      const uint32_t sel = (x ^ s1) & 3u;
      own = (v >> (sel << 3)) & 0xFFu;
      other = (v >> ((sel ^ 1u) << 3)) & 0xFFu;
    } else {
      const uint32_t r = __funnelshift_l(v, v, ((x ^ s1) & 1u) << 4);
      own = r & 0xFFFFu;
      other = r >> 16;
    }
  }
}

// Second pass: every endpoint of the window, and the pivot, get the endpoint's
// Lemma 1 totals. A thread takes whole counter words, most of which hold no
// endpoint in a butterfly (an endpoint is in one from two wedges on).
template <int CW>
__device__ __forceinline__ void credit_window(const uint32_t* words, const Win& w, uint32_t wlo, uint32_t whi,
                                              int64_t end_base, const TipOut& o, uint64_t& pb, uint64_t& pu) {
  auto endpoint = [&](uint32_t rank, uint32_t p, uint32_t q) {
    if (p + q < 2u) return;
    uint64_t eb, eu;
    if (CW <= 8) {
      eb = (p * (p - (p > 0u)) + q * (q - (q > 0u))) >> 1;
      eu = p * q;
    } else {
      eb = eu = 0;
      endpoint_contrib(((unsigned long long)q << 32) | p, eb, eu);
    }
    add_vertex(o, end_base + rank, eb, eu);
    pb += eb;
    pu += eu;
  };
  if constexpr (CW == 32) {
    for (uint32_t k = threadIdx.x; k < whi - wlo; k += kSweepThreads) endpoint(wlo + k, words[2 * k],
                                                                               words[2 * k + 1]);
  } else {
    const uint32_t first = CW == 4 ? wlo & ~3u : CW == 8 ? wlo & ~1u : wlo;  // rank of word 0's first counter
    for (uint32_t k = threadIdx.x; k < w.words; k += kSweepThreads) {
      const uint32_t v = words[k];
      if (v == 0u) continue;
      if constexpr (CW == 16) {
        endpoint(first + k, v & 0xFFFFu, v >> 16);
      } else if constexpr (CW == 8) {
        endpoint(first + 2 * k, v & 0xFFu, (v >> 8) & 0xFFu);
        endpoint(first + 2 * k + 1, (v >> 16) & 0xFFu, v >> 24);
      } else {
#pragma unroll
        for (int j = 0; j < 4; j++) endpoint(first + 4 * k + j, (v >> (8 * j)) & 0xFu, (v >> (8 * j + 4)) & 0xFu);
      }
    }
  }
}

// First pass: count all L neighbours' entries in the window; every neighbour
// that has some moves its slot past them and joins the segment list.
template <int G, int CW>
__device__ __forceinline__ void tips_count(const CsrView& g, const PivotGeom& q, uint2* slots, uint32_t* next,
                                           Segment* seg, uint32_t* n_seg, const Win& w) {
  const int gl = threadIdx.x & (G - 1);
  uint64_t unused_b = 0, unused_u = 0;
  SlotBatch sb;
  LaneBatch b;
  slot_fetch<G>(slots, q.L, next, sb);
  batch_load<G>(g.col, sb, b);
  while (b.base < q.L) {  // warp-uniform
    const uint32_t i = b.base + lane_id() / G;
    const uint32_t en = b.e.x + (b.e.y & 0x7FFFFFFFu);
    uint32_t cn, xn;
    if (lean_walk<G, CW, false>(g.col, b.e.x, en, b.e.y >> 31, b.x, w, gl, i < q.L, unused_b, unused_u, cn, xn) &&
        i < q.L && cn != b.e.x) {
      slots[i] = lean_slot(cn, en, b.e.y >> 31);
      const uint32_t k = atomicAdd(n_seg, 1u);
      if (DBBC_CHECK(k < q.L)) seg[k] = Segment{b.e.x, cn, g.col[q.rb + i], i};
    }
    __syncwarp();
    slot_fetch<G>(slots, q.L, next, sb);
    batch_load<G>(g.col, sb, b);
  }
}

// Last pass: walk the n listed segments again. A wedge with own-class count p
// and other-class count q is in p - 1 balanced and q unbalanced butterflies.
// Sums of one segment fit 32 bits in the narrow widths (see lean_walk).
template <int G, int CW, bool VERT, bool EDGE>
__device__ __forceinline__ void tips_credit(const CsrView& g, const PivotGeom& q, const Segment* seg, uint32_t n,
                                            uint32_t* next, const Win& w, const TipOut& o) {
  using Sum = typename std::conditional<CW == 32, uint64_t, uint32_t>::type;
  const uint32_t gl = threadIdx.x & (G - 1);
  for (;;) {
    uint32_t base = 0;
    if (lane_id() == 0) base = atomicAdd(next, 32u / G);
    base = __shfl_sync(kFullMask, base, 0);
    if (base >= n) break;  // warp-uniform
    const uint32_t k = base + lane_id() / G;
    Segment t{0u, 0u, 0u, 0u};
    if (k < n) t = seg[k];
    const uint32_t s1 = t.e & 1u, len = t.end - t.c, start = t.c & ~3u;
    const uint32_t chunks = (t.end - start + 4u * G - 1u) / (4u * G);
    const uint32_t trips = __reduce_max_sync(kFullMask, chunks);
    Sum sb = 0, su = 0;
    // Edges: the group's lanes take consecutive entries, so that the adds to
    // the far edges of G lanes fall into G / 4 sectors (four entries per lane
    // would spread them over G sectors: 28.5 instead of 19.8 ms of sweep on the
    // 20M-edge rating graph). Vertices: four entries per lane by one load.
    constexpr uint32_t kLane = EDGE ? 1u : 4u, kItem = EDGE ? (uint32_t)G : 1u;
    auto load = [&](uint32_t pos, uint32_t (&x)[kLU]) {
      if constexpr (EDGE) {
#pragma unroll
        for (int u = 0; u < kLU; u++) x[u] = pos + u * kItem < t.end ? __ldg(g.col + pos + u * kItem) : 0u;
      } else {
        x[0] = x[1] = x[2] = x[3] = 0u;
        if (pos < t.end) lean_load(g.col, pos, x);
      }
    };
    uint32_t pos = start + gl * kLane;
    uint32_t x[kLU];
    load(pos, x);
    for (uint32_t j = 0; j < trips; j++, pos += 4u * G) {
      uint32_t y[kLU];
      load(pos + 4u * G, y);  // the next chunk, while this one is credited
#pragma unroll
      for (int u = 0; u < kLU; u++) {
        if (pos + u * kItem - t.c < len) {
          uint32_t own, other;
          counter_pair<CW>(x[u], s1, w, own, other);
          if (EDGE) add_edge(o, pos + u * kItem, own - 1u, other);
          sb += own - 1u;
          su += other;
        }
        x[u] = y[u];
      }
    }
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) {  // sum over the group's lanes
      sb += __shfl_xor_sync(kFullMask, sb, off);
      su += __shfl_xor_sync(kFullMask, su, off);
    }
    if (k < n && gl == 0) {
      if (VERT) add_vertex(o, q.base + (t.e >> 1), sb, su);
      if (EDGE) add_edge(o, q.rb + t.i, sb, su);
    }
  }
}

// Block-uniform counters of the window being swept, in shared memory.
struct TipsShared {
  uint32_t next_count, next_credit, n_seg;
};

template <int G, int CW, bool VERT, bool EDGE>
__device__ __forceinline__ void tips_window(const CsrView& g, const PivotGeom& q, uint2* slots, Segment* seg,
                                            TipsShared& sh, uint32_t lo, uint32_t hi, uint32_t sbase, uint32_t* words,
                                            const TipOut& o, uint64_t& pb, uint64_t& pu) {
  const Win w = make_win(CW, lo, hi, sbase);
  tips_count<G, CW>(g, q, slots, &sh.next_count, seg, &sh.n_seg, w);
  __syncthreads();
  if (VERT) {
    credit_window<CW>(words, w, lo, hi, q.base == 0 ? (int64_t)g.n_u : 0, o, pb,
                      pu);  // endpoints share the pivot's side
  }
  const uint32_t n = DBBC_CHECK(sh.n_seg <= q.L) ? sh.n_seg : q.L;
  tips_credit<G, CW, VERT, EDGE>(g, q, seg, n, &sh.next_credit, w, o);
  __syncthreads();
  zero_words(words, w.words);
  if (threadIdx.x == 0) sh = TipsShared{0u, 0u, 0u};
  __syncthreads();
}

template <int CW, bool VERT, bool EDGE, typename... A>
__device__ __forceinline__ void tips_window_dispatch(int group_log, A&&... a) {
  switch (group_log) {
    case 0: tips_window<1, CW, VERT, EDGE>(a...); break;
    case 2: tips_window<4, CW, VERT, EDGE>(a...); break;
    case 3: tips_window<8, CW, VERT, EDGE>(a...); break;
    case 4: tips_window<16, CW, VERT, EDGE>(a...); break;
    default: tips_window<32, CW, VERT, EDGE>(a...); break;
  }
}

// Per CTA: cur_cap neighbour slots and cur_cap segments of scratch.
template <bool VERT, bool EDGE>
__global__ void __launch_bounds__(kSweepThreads, 1) tips_sweep_kernel(CsrView g, const SweepItem* __restrict__ items,
                                                                   int64_t n_items, int* next_item,
                                                                   uint2* __restrict__ cursors,
                                                                   Segment* __restrict__ segments, int64_t cur_cap,
                                                                   TipOut o) {
  extern __shared__ __align__(16) unsigned char sweep_smem[];
  uint32_t* words = reinterpret_cast<uint32_t*>(sweep_smem);
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(sweep_smem);
  __shared__ int item_sh;
  __shared__ TipsShared sh;
  __shared__ unsigned long long red[2][kSweepThreads / 32];
  const int tid = threadIdx.x;
  zero_words(words, kSweepWords);
  if (tid == 0) sh = TipsShared{0u, 0u, 0u};
  uint2* cur = cursors + (int64_t)blockIdx.x * cur_cap;
  Segment* seg = segments + (int64_t)blockIdx.x * cur_cap;
  for (;;) {
    if (tid == 0) item_sh = atomicAdd(next_item, 1);
    __syncthreads();
    const int64_t it = item_sh;
    __syncthreads();
    if (it >= n_items) break;
    const SweepItem item = items[it];
    PivotGeom q = pivot_geom(g, item.row);
    if (!DBBC_CHECK((int64_t)q.L <= cur_cap)) q.L = 0;  // checked builds: cursor capacity
    const ItemWindows iw(item);
    for (uint32_t i = tid; i < q.L; i += kSweepThreads) {
      uint32_t b, en, s1;
      lean_cursor_start(g, q, i, (item.flags & kItemFirst) ? 0u : item.lo, b, en, s1);
      cur[i] = lean_slot(b, en, s1);
    }
    __syncthreads();
    uint64_t pb = 0, pu = 0;
    for (uint32_t r = 0; r < iw.count(); r++) {
      uint32_t lo, hi;
      int cw;
      iw.window(r, lo, hi, cw);
      const int gl = item.group_log;
      if (cw == 4) tips_window_dispatch<4, VERT, EDGE>(gl, g, q, cur, seg, sh, lo, hi, sbase, words, o, pb, pu);
      else if (cw == 8) tips_window_dispatch<8, VERT, EDGE>(gl, g, q, cur, seg, sh, lo, hi, sbase, words, o, pb, pu);
      else if (cw == 16) tips_window_dispatch<16, VERT, EDGE>(gl, g, q, cur, seg, sh, lo, hi, sbase, words, o, pb, pu);
      else tips_window_dispatch<32, VERT, EDGE>(gl, g, q, cur, seg, sh, lo, hi, sbase, words, o, pb, pu);
    }
    if (VERT) {  // the pivot's share of this item
      pb = warp_sum_u64(pb);
      pu = warp_sum_u64(pu);
      if (lane_id() == 0) {
        red[0][tid >> 5] = pb;
        red[1][tid >> 5] = pu;
      }
      __syncthreads();
      if (tid < 32) {
        uint64_t x = tid < kSweepThreads / 32 ? red[0][tid] : 0, y = tid < kSweepThreads / 32 ? red[1][tid] : 0;
        x = warp_sum_u64(x);
        y = warp_sum_u64(y);
        if (tid == 0) add_vertex(o, item.row, x, y);
      }
      __syncthreads();
    }
  }
}

__global__ void rows_to_ids_kernel(const int32_t* __restrict__ vertex, int64_t n, const unsigned long long* rb,
                                   const unsigned long long* ru, unsigned long long* ob, unsigned long long* ou) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    ob[vertex[r]] = rb[r];
    ou[vertex[r]] = ru[r];
  }
}

__global__ void row_of_id_kernel(const int32_t* __restrict__ vertex, int64_t n, int32_t* __restrict__ row_of) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
    row_of[vertex[r]] = (int32_t)r;
}

// Position in [b, e) of a row whose entry has side rank r, or -1 (rows are
// sorted by entry, and an entry is (side rank << 1) | negative).
__device__ __forceinline__ int64_t find_in_row(const uint32_t* col, int64_t b, int64_t e, uint32_t r) {
  const uint32_t key = r << 1;
  const int64_t end = e;
  while (b < e) {
    const int64_t mid = (b + e) >> 1;
    if (col[mid] < key) b = mid + 1; else e = mid;
  }
  return b < end && (col[b] >> 1) == r ? b : -1;
}

// Per queried pair (U id, V id): the sum of the counts at the edge's two CSR
// positions, or zeros when the pair is not an edge; ids out of range set err.
__global__ void edge_query_kernel(CsrView g, const int32_t* __restrict__ row_of, const int32_t* __restrict__ qu,
                                  const int32_t* __restrict__ qv, int64_t k, const unsigned long long* eb,
                                  const unsigned long long* eu, unsigned long long* ob, unsigned long long* ou,
                                  unsigned* err) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < k; i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = qu[i], b = qv[i];
    unsigned long long xb = 0, xu = 0;
    if (a < 0 || a >= g.n_u || b < 0 || (int64_t)b >= g.n - g.n_u) {
      atomicOr(err, 1u);
    } else {
      const int64_t ru = row_of[a], rv = row_of[(int64_t)g.n_u + b];
      const int64_t p1 = find_in_row(g.col, g.row_ptr[ru], g.row_ptr[ru + 1], (uint32_t)(rv - g.n_u));
      const int64_t p2 = find_in_row(g.col, g.row_ptr[rv], g.row_ptr[rv + 1], (uint32_t)ru);
      if (p1 >= 0 && p2 >= 0) {
        xb = eb[p1] + eb[p2];
        if (eu) {
          xu = eu[p1] + eu[p2];
        } else {  // both counts in one word, each below 2^32
          xu = xb >> 32;
          xb &= 0xFFFFFFFFull;
        }
      }
    }
    ob[i] = xb;
    ou[i] = xu;
  }
}

template <bool VERT, bool EDGE>
void enqueue_tips(const dbbc_graph* g, cudaStream_t s, const TipOut& o, unsigned* d_status, Scratch& sc) {
  if (g->n_piv == 0) return;
  const CsrView view{g->row_ptr, g->span, g->col, g->lower, g->n_u, g->n, g->nnz};
  const int sms = num_sms();
  if (g->n_light > 0) {
    auto fn = tips_light_kernel<VERT, EDGE>;
    const int slots_log = tier_slots_log(g->tune.light_max_work, g->tune.hash_mult_log, 10);
    const size_t smem = (size_t)kLightWarps * ((size_t)1 << slots_log) * kHashSlotBytes;
    const int64_t want = ceil_div<int64_t>(g->n_light, kLightWarps);
    const int64_t cap = (int64_t)sms * resident_ctas((const void*)fn, kLightWarps * 32, smem,
                                                     (size_t)kLightWarps * kLightSlots * kHashSlotBytes);
    fn<<<(unsigned)std::min(want, cap), kLightWarps * 32, smem, s>>>(
        view, g->order + g->n_hub + g->n_medium, g->work, g->n_light, g->tune.hash_mult_log, slots_log, o, d_status);
    DBBC_LAUNCH_CHECK();
  }
  if (g->n_medium > 0) {
    auto fn = tips_medium_kernel<VERT, EDGE>;
    const int slots_log = tier_slots_log(g->tune.medium_max_work, g->tune.hash_mult_log, 13);
    const size_t smem = ((size_t)1 << slots_log) * kHashSlotBytes;
    const int64_t cap = (int64_t)sms * resident_ctas((const void*)fn, kMediumThreads, smem,
                                                     (size_t)kMediumSlots * kHashSlotBytes);
    fn<<<(unsigned)std::min<int64_t>(g->n_medium, cap), kMediumThreads, smem, s>>>(
        view, g->order + g->n_hub, g->work, g->n_medium, g->tune.hash_mult_log, slots_log, o, d_status);
    DBBC_LAUNCH_CHECK();
  }
  if (g->n_hub > 0) {
    auto fn = tips_sweep_kernel<VERT, EDGE>;
    const size_t smem = kSweepSmem;
    const int grid = sms * resident_ctas((const void*)fn, kSweepThreads, smem, smem);
    uint2* cursors = sc.get<uint2>((size_t)grid * (size_t)g->sweep_max_lower);
    Segment* segments = sc.get<Segment>((size_t)grid * (size_t)g->sweep_max_lower);
    int* next = sc.get<int>(1);
    DBBC_CUDA(cudaMemsetAsync(next, 0, sizeof(int), s));
    fn<<<grid, kSweepThreads, smem, s>>>(view, g->sweep_items, g->n_sweep_items, next, cursors, segments,
                                         g->sweep_max_lower, o);
    DBBC_LAUNCH_CHECK();
  }
}

inline unsigned grid_1d(int64_t n) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 4096));
}

}  // namespace dbbc

using namespace dbbc;

extern "C" dbbc_status dbbc_count_vertices(const dbbc_graph* g, void* cuda_stream, uint64_t* balanced_v,
                                           uint64_t* unbalanced_v) {
  if (!g || (g->n > 0 && (!balanced_v || !unbalanced_v))) return DBBC_EINVAL;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  try {
    if (g->n == 0) return DBBC_OK;
    Scratch sc(s);
    const int64_t n = g->n;
    unsigned long long* rows = sc.get<unsigned long long>((size_t)(4 * n));  // row sums, then per-id output
    unsigned* d_status = sc.get<unsigned>(1);
    DBBC_CUDA(cudaMemsetAsync(rows, 0, (size_t)(2 * n) * 8, s));
    DBBC_CUDA(cudaMemsetAsync(d_status, 0, sizeof(unsigned), s));
    TipOut o;
    o.vb = rows;
    o.vu = rows + n;
    o.n = n;
    enqueue_tips<true, false>(g, s, o, d_status, sc);
    unsigned long long* ob = rows + 2 * n;
    unsigned long long* ou = rows + 3 * n;
    rows_to_ids_kernel<<<grid_1d(n), 256, 0, s>>>(g->vertex, n, o.vb, o.vu, ob, ou);
    DBBC_LAUNCH_CHECK();
    DBBC_CUDA(cudaMemcpyAsync(balanced_v, ob, (size_t)n * 8, cudaMemcpyDeviceToHost, s));
    DBBC_CUDA(cudaMemcpyAsync(unbalanced_v, ou, (size_t)n * 8, cudaMemcpyDeviceToHost, s));
    unsigned h = 0;
    DBBC_CUDA(cudaMemcpyAsync(&h, d_status, sizeof(h), cudaMemcpyDeviceToHost, s));
    DBBC_CUDA(cudaStreamSynchronize(s));
    raise_device_status(h);
  } catch (const Error& e) {
    return e.status;
  } catch (...) {
    return DBBC_EINTERNAL;
  }
  return DBBC_OK;
}

extern "C" dbbc_status dbbc_count_edges(const dbbc_graph* g, void* cuda_stream, const int32_t* qu, const int32_t* qv,
                                        int64_t k, uint32_t flags, uint64_t* balanced_e, uint64_t* unbalanced_e) {
  if (!g || k < 0 || (flags & ~(uint32_t)DBBC_INPUT_DEVICE) != 0) return DBBC_EINVAL;
  if (k == 0) return DBBC_OK;
  if (!qu || !qv || !balanced_e || !unbalanced_e) return DBBC_EINVAL;
  if (g->n_u == 0 || g->n == g->n_u) return DBBC_EINVAL;  // no pair is in range
  const bool on_device = (flags & DBBC_INPUT_DEVICE) != 0;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  try {
    Scratch sc(s);
    const int64_t n = g->n, nnz = g->nnz;
    // an edge (u, v) is in at most (deg(u) - 1)(deg(v) - 1) butterflies: when
    // that fits 32 bits for the largest degrees, both counts share a word
    const size_t words = (uint64_t)g->max_deg_u * (uint64_t)g->max_deg_v >> 32 ? 2 : 1;
    unsigned long long* acc = sc.get<unsigned long long>(words * (size_t)nnz);
    unsigned* d_status = sc.get<unsigned>(2);  // [0] device checks, [1] ids out of range
    int32_t* row_of = sc.get<int32_t>((size_t)n);
    DBBC_CUDA(cudaMemsetAsync(acc, 0, words * (size_t)nnz * 8, s));
    DBBC_CUDA(cudaMemsetAsync(d_status, 0, 2 * sizeof(unsigned), s));
    TipOut o;
    o.eb = acc;
    o.eu = words == 2 ? acc + nnz : nullptr;
    o.nnz = nnz;
    enqueue_tips<false, true>(g, s, o, d_status, sc);
    row_of_id_kernel<<<grid_1d(n), 256, 0, s>>>(g->vertex, n, row_of);
    DBBC_LAUNCH_CHECK();
    const int32_t* dqu = qu;
    const int32_t* dqv = qv;
    unsigned long long* ob = reinterpret_cast<unsigned long long*>(balanced_e);
    unsigned long long* ou = reinterpret_cast<unsigned long long*>(unbalanced_e);
    if (!on_device) {
      int32_t* q = sc.get<int32_t>((size_t)(2 * k));
      DBBC_CUDA(cudaMemcpyAsync(q, qu, (size_t)k * 4, cudaMemcpyHostToDevice, s));
      DBBC_CUDA(cudaMemcpyAsync(q + k, qv, (size_t)k * 4, cudaMemcpyHostToDevice, s));
      dqu = q;
      dqv = q + k;
      ob = sc.get<unsigned long long>((size_t)(2 * k));
      ou = ob + k;
    }
    const CsrView view{g->row_ptr, g->span, g->col, g->lower, g->n_u, g->n, g->nnz};
    edge_query_kernel<<<grid_1d(k), 256, 0, s>>>(view, row_of, dqu, dqv, k, o.eb, o.eu, ob, ou, d_status + 1);
    DBBC_LAUNCH_CHECK();
    if (!on_device) {
      DBBC_CUDA(cudaMemcpyAsync(balanced_e, ob, (size_t)k * 8, cudaMemcpyDeviceToHost, s));
      DBBC_CUDA(cudaMemcpyAsync(unbalanced_e, ou, (size_t)k * 8, cudaMemcpyDeviceToHost, s));
    }
    unsigned h[2] = {0, 0};
    DBBC_CUDA(cudaMemcpyAsync(h, d_status, sizeof(h), cudaMemcpyDeviceToHost, s));
    DBBC_CUDA(cudaStreamSynchronize(s));
    if (h[1]) return DBBC_EINVAL;
    raise_device_status(h[0]);
  } catch (const Error& e) {
    return e.status;
  } catch (...) {
    return DBBC_EINTERNAL;
  }
  return DBBC_OK;
}
