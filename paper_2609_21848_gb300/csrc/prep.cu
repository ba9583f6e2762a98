// Graph build on the device: validate, keep-latest deduplication, degrees,
// Def. 3 priority ranks, sign-packed CSR sorted by priority, accepted-wedge
// work per pivot (Algorithm 1's inner loop bounds), and the counting tiers.
#include <algorithm>
#include <cstring>

#include "internal.h"
#include "radix.cuh"

namespace dbbc {

// Components of a disjoint union as seen by the kernels: component c owns the
// side ids (and, after ranking, the side ranks) [uo(c), uo(c + 1)) of U and
// [vo(c), vo(c + 1)) of V. A plain graph is one component and has no arrays.
__device__ __forceinline__ int32_t component_of(const int64_t* off, int32_t n_graphs, int64_t side_id);
struct UnionView {
  const int64_t* uoff;
  const int64_t* voff;
  int32_t n_graphs;
  int64_t n_u, n_v;
  __device__ __forceinline__ int64_t uo(int32_t c) const { return n_graphs == 1 ? (c ? n_u : 0) : uoff[c]; }
  __device__ __forceinline__ int64_t vo(int32_t c) const { return n_graphs == 1 ? (c ? n_v : 0) : voff[c]; }
  __device__ __forceinline__ int32_t comp_u(int64_t id) const {
    return n_graphs == 1 ? 0 : component_of(uoff, n_graphs, id);
  }
  __device__ __forceinline__ int32_t comp_v(int64_t id) const {
    return n_graphs == 1 ? 0 : component_of(voff, n_graphs, id);
  }
};

__device__ __forceinline__ int32_t component_of(const int64_t* off, int32_t n_graphs, int64_t side_id) {
  int64_t lo = 0, hi = (int64_t)n_graphs + 1;  // upper_bound over off[0 .. n_graphs]
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (off[mid] <= side_id) lo = mid + 1; else hi = mid;
  }
  return (int32_t)(lo - 1);
}

// ------------------------------------------------------------------ kernels
template <typename T>
__device__ __forceinline__ int64_t lower_bound_dev(const T* a, int64_t n, T x) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (a[mid] < x) lo = mid + 1; else hi = mid;
  }
  return lo;
}
template <typename T>
__device__ __forceinline__ int64_t upper_bound_dev(const T* a, int64_t n, T x) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (a[mid] <= x) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// deg[id] += 1 for every lane with ok, as one atomic per run of equal ids in
// consecutive lanes (edges that arrive grouped by an endpoint form long runs).
__device__ __forceinline__ void add_runs(int32_t* __restrict__ deg, int32_t id, bool ok) {
  const unsigned lane = lane_id();
  const int32_t x = ok ? id : -1;
  const int32_t prev = __shfl_up_sync(kFullMask, x, 1);
  const bool head = lane == 0 || prev != x;
  const unsigned heads = __ballot_sync(kFullMask, head);
  const unsigned later = lane == 31 ? 0u : heads & (~0u << (lane + 1));
  const int len = (later ? __ffs(later) - 1 : 32) - (int)lane;
  if (ok && head) atomicAdd(&deg[x], len);
}

// Validation and degrees in one read of the edges: flags the edges whose ids
// are out of range or whose sign is not +-1 (every later kernel of the build
// then returns at once), and counts the others' degrees over unified ids (V
// ids follow the U ids).
__global__ void degree_kernel(const int32_t* __restrict__ eu, const int32_t* __restrict__ ev,
                              const int8_t* __restrict__ es, int64_t m, int32_t n_u, int32_t n_v,
                              int32_t* __restrict__ deg, unsigned* flags) {
  constexpr int kRound = 4;  // edges per thread per round, their loads in flight together
  let_next_start();
  wait_for_previous();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t iters = (m + stride - 1) / stride;  // the same for every lane: the warp votes together
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned bad = 0;
  for (int64_t it = 0; it < iters; it += kRound) {
    int32_t a[kRound], b[kRound];
    int8_t c[kRound];
#pragma unroll
    for (int j = 0; j < kRound; j++) {
      const int64_t i = (it + j) * stride + t0;
      a[j] = i < m ? eu[i] : 0;
      b[j] = i < m ? ev[i] : 0;
      c[j] = i < m ? es[i] : (int8_t)1;
    }
#pragma unroll
    for (int j = 0; j < kRound; j++) {
      const bool in = (it + j) * stride + t0 < m;
      const bool ok_u = a[j] >= 0 && a[j] < n_u, ok_v = b[j] >= 0 && b[j] < n_v;
      if (in) bad |= (ok_u ? 0u : kPrepBadU) | (ok_v ? 0u : kPrepBadV) | (c[j] == 1 || c[j] == -1 ? 0u : kPrepBadSign);
      add_runs(deg, a[j], in && ok_u);
      add_runs(deg, ok_v ? n_u + b[j] : 0, in && ok_v);
    }
  }
  bad = __reduce_or_sync(kFullMask, bad);
  if (lane_id() == 0 && bad) atomicOr(flags, bad);
}

// Sort key per vertex: (side, component, degree, id within the component).
// Ascending order is the Def. 3 priority within each side of each component
// (V ids follow U ids in the unified space); components occupy contiguous
// rank ranges, which keeps a component's accepted endpoints together.
// Degrees of distinct edges fit bits_deg; repeated pairs can push one past it,
// and is cut off there: such a list is ranked again without the repeats.
// Counts the digits of the sort (bits_id and up) as it goes.
__global__ void __launch_bounds__(256) vertex_keys_kernel(const int32_t* __restrict__ deg, int64_t n, int32_t n_u,
                                                          int bits_comp, int bits_deg, int bits_id, UnionView un,
                                                          uint64_t* __restrict__ key, int passes, uint32_t* hist,
                                                          const unsigned* flags) {
  __shared__ uint32_t h[kRsMaxPasses][256];
  if (cta_stopped(flags)) return;
  DigitCounts dc{h, passes, bits_id};
  dc.start();
  const uint64_t deg_mask = (1ull << bits_deg) - 1;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t side = x >= n_u ? 1 : 0;
    const int64_t sid = side ? x - n_u : x;
    const int32_t c = side ? un.comp_v(sid) : un.comp_u(sid);
    const uint64_t local = (uint64_t)(sid - (side ? un.vo(c) : un.uo(c)));
    const uint64_t k = (side << (bits_comp + bits_deg + bits_id)) | ((uint64_t)c << (bits_deg + bits_id)) |
                       (min((uint64_t)(uint32_t)deg[x], deg_mask) << bits_id) | local;
    key[x] = k;
    dc.add(k);
  }
  dc.finish(hist);
}

// Rows in rank order: vertex, degree and (unions) component of every row, the
// rank of every vertex, and the row pointers, whose prefix sum runs in the
// same kernel over tiles of kRowTile rows (tile_prefix). Clears the rows' work.
constexpr int kRowThreads = 256;
constexpr int kRowItems = 4;
constexpr int kRowTile = kRowThreads * kRowItems;

__global__ void __launch_bounds__(kRowThreads) ranks_kernel(const uint64_t* __restrict__ skey, int64_t n, int32_t n_u,
                                                            int bits_comp, int bits_deg, int bits_id, UnionView un,
                                                            int32_t* __restrict__ vertex,
                                                            int32_t* __restrict__ side_rank,
                                                            int32_t* __restrict__ rowdeg,
                                                            int64_t* __restrict__ row_ptr,
                                                            int32_t* __restrict__ component,
                                                            uint64_t* __restrict__ work, int64_t* lone,
                                                            uint64_t* state, unsigned* counter, unsigned* flags) {
  __shared__ uint64_t tot_sh;
  const int64_t tile = take_tile(counter, flags);
  if (tile < 0) return;
  const uint64_t id_mask = (1ull << bits_id) - 1, deg_mask = (1ull << bits_deg) - 1;
  const uint64_t comp_mask = (1ull << bits_comp) - 1;
  const int64_t r0 = tile * kRowTile + (int64_t)threadIdx.x * kRowItems;
  uint32_t d[kRowItems];
  uint64_t sum = 0;
#pragma unroll
  for (int j = 0; j < kRowItems; j++) {
    const int64_t r = r0 + j;
    d[j] = 0;
    if (r < n) {
      const uint64_t k = skey[r];
      const bool side = (k >> (bits_comp + bits_deg + bits_id)) & 1;
      const int32_t c = bits_comp ? (int32_t)((k >> (bits_deg + bits_id)) & comp_mask) : 0;
      const int64_t local = (int64_t)(k & id_mask);
      const int32_t x = side ? (int32_t)(n_u + un.vo(c) + local) : (int32_t)(un.uo(c) + local);
      d[j] = (uint32_t)((k >> bits_id) & deg_mask);
      if (d[j] < 2u && un.n_graphs == 1) {  // the side's last one sets the side's count
        const int64_t end = side ? n : n_u;
        if (r + 1 == end || ((skey[r + 1] >> bits_id) & deg_mask) >= 2u) lone[side] = r + 1 - (side ? n_u : 0);
      }
      if (DBBC_CHECK(x >= 0 && x < n)) {
        vertex[r] = x;
        side_rank[x] = side ? (int32_t)(r - n_u) : (int32_t)r;
        rowdeg[r] = (int32_t)d[j];
        work[r] = 0;
        if (component) component[r] = c;
      }
    }
    sum += d[j];
  }
  uint64_t run = block_excl_scan<uint64_t, kRowThreads>(sum, &tot_sh);
  __syncthreads();
  uint64_t prefix;
  if (!tile_prefix(state, tile, tot_sh, flags, &prefix)) return;
  run += prefix;
#pragma unroll
  for (int j = 0; j < kRowItems; j++) {
    const int64_t r = r0 + j;
    if (r < n) row_ptr[r] = (int64_t)run;
    run += d[j];
    if (r == n - 1) row_ptr[n] = (int64_t)run;
  }
}

// CSR keys in two sorts. The U rows are the edges sorted by
// ku = (U rank << (bits_v + 1)) | (V rank << 1) | negative; the V rows are the
// same list re-sorted stably by V rank alone, as
// kv = (V rank << (bits_u + 1)) | (U rank << 1) | negative, which keeps every
// V row ascending by U rank. The last pass of each sort also writes the rows'
// entries (the low bits of the key).
__global__ void __launch_bounds__(256) csr_u_keys_kernel(const int32_t* __restrict__ eu,
                                                         const int32_t* __restrict__ ev,
                                                         const int8_t* __restrict__ es, int64_t m, int32_t n_u,
                                                         const int32_t* __restrict__ side_rank, int bits_v,
                                                         uint64_t* __restrict__ ku, int passes, uint32_t* hist,
                                                         const unsigned* flags) {
  __shared__ uint32_t h[kRsMaxPasses][256];
  if (cta_stopped(flags)) return;
  DigitCounts dc{h, passes, 1};
  dc.start();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t ru = (uint32_t)side_rank[eu[i]];
    const uint64_t rv = (uint32_t)side_rank[n_u + ev[i]];
    const uint64_t k = (ru << (bits_v + 1)) | (rv << 1) | (es[i] < 0 ? 1u : 0u);
    ku[i] = k;
    dc.add(k);
  }
  dc.finish(hist);
}

// V key of a U key.
struct VKey {
  int bits_u, bits_v;
  __device__ __forceinline__ uint64_t operator()(uint64_t k) const {
    const uint64_t ru = k >> (bits_v + 1), rv = (k >> 1) & ((1ull << bits_v) - 1);
    return (rv << (bits_u + 1)) | (ru << 1) | (k & 1u);
  }
};

// The first pass of the V sort reads the U-sorted list: V keys, each with its
// U position (the edge's position in its U row) as the value.
struct VKeyLoad {
  const uint64_t* ku;
  VKey vk;
  __device__ __forceinline__ uint64_t key(uint32_t i) const { return vk(ku[i]); }
  __device__ __forceinline__ uint32_t val(uint32_t i) const { return i; }
};

// Flags a repeated (u, v) pair (U-sorted keys that agree in everything but the
// sign bit are adjacent) and counts the digits of the V sort.
__global__ void __launch_bounds__(256) csr_v_digits_kernel(const uint64_t* __restrict__ ku, int64_t m, VKey vk,
                                                           int passes, uint32_t* hist, unsigned* flags) {
  __shared__ uint32_t h[kRsMaxPasses][256];
  if (cta_stopped(flags)) return;
  DigitCounts dc{h, passes, 1 + vk.bits_u};
  dc.start();
  bool dup = false;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = ku[i];
    if (i + 1 < m) dup |= (k >> 1) == (ku[i + 1] >> 1);
    dc.add(vk(k));
  }
  if (__syncthreads_or(dup)) {
    if (threadIdx.x == 0) atomicOr(flags, (unsigned)kPrepDup);
    return;
  }
  dc.finish(hist);
}

// The distinct edges of a U-sorted list with repeated pairs: the last of every
// run (the sorts are stable, so the latest input occurrence), compacted in one
// pass over tiles of kRowTile edges. *count gets their number.
__global__ void __launch_bounds__(kRowThreads) dedup_kernel(const uint64_t* __restrict__ ku, int64_t m, int bits_v,
                                                            int32_t n_u, int64_t n,
                                                            const int32_t* __restrict__ vertex,
                                                            int32_t* __restrict__ eu, int32_t* __restrict__ ev,
                                                            int8_t* __restrict__ es, uint64_t* count, uint64_t* state,
                                                            unsigned* counter, unsigned* flags) {
  __shared__ uint32_t tot_sh;
  const int64_t tile = take_tile(counter, flags);
  if (tile < 0) return;
  const int64_t i0 = tile * kRowTile + (int64_t)threadIdx.x * kRowItems;
  uint64_t k[kRowItems + 1];
#pragma unroll
  for (int j = 0; j <= kRowItems; j++) k[j] = i0 + j < m ? ku[i0 + j] : ~0ull;
  bool keep[kRowItems];
  uint32_t sum = 0;
#pragma unroll
  for (int j = 0; j < kRowItems; j++) {
    keep[j] = i0 + j < m && (i0 + j == m - 1 || (k[j] >> 1) != (k[j + 1] >> 1));
    sum += keep[j] ? 1u : 0u;
  }
  const uint32_t ex = block_excl_scan<uint32_t, kRowThreads>(sum, &tot_sh);
  __syncthreads();
  uint64_t prefix;
  if (!tile_prefix(state, tile, tot_sh, flags, &prefix)) return;
  uint64_t at = prefix + ex;
#pragma unroll
  for (int j = 0; j < kRowItems; j++) {
    if (keep[j]) {
      const uint64_t ru = k[j] >> (bits_v + 1), rv = (k[j] >> 1) & ((1ull << bits_v) - 1);
      if (DBBC_CHECK(at < (uint64_t)m && ru < (uint64_t)n_u && (int64_t)(n_u + rv) < n)) {
        eu[at] = vertex[ru];
        ev[at] = vertex[n_u + rv] - n_u;
        es[at] = (k[j] & 1u) ? (int8_t)-1 : (int8_t)1;
      }
      at++;
    }
    if (i0 + j == m - 1) *count = at;
  }
}

// V keys and U positions of the V rows: the edge at V position m + k.
struct CsrKeys {
  const uint64_t* kv;
  const uint32_t* upos;
  int64_t m;
  int32_t n_u;
  int bits_u;
};

// lower[r] = neighbours of row r with lower Def. 3 priority. A U vertex of
// degree d is above a V vertex iff deg(v) < d (equal degree: the V id is
// larger); a V vertex of degree d is above a U vertex iff deg(u) <= d.
// Neighbours lie in the row's own component, whose other-side ranks ascend by
// degree, and rows list neighbours by ascending side rank, so the lower ones
// are a prefix.
// The last CTA instead finds, per side, how many vertices have degree below
// each of four limits (ranks ascend by degree within a side): below[2k] for U,
// below[2k + 1] for V; and the largest degree, that of some component's last
// rank. Also writes the rows' spans (see CsrView).
struct DegreeLimits {
  int32_t d[4];
};
__global__ void lower_kernel(const int64_t* __restrict__ row_ptr, const uint32_t* __restrict__ col,
                             const int32_t* __restrict__ rowdeg, int64_t n, int32_t n_u, UnionView un,
                             uint32_t* __restrict__ lower, uint2* __restrict__ span, const int64_t* lone,
                             DegreeLimits lim, int64_t* below,
                             unsigned* max_deg, const unsigned* flags) {
  if (cta_stopped(flags)) return;
  if (blockIdx.x == gridDim.x - 1) {
    const int t = threadIdx.x;
    if (t < 8) {
      const bool u = (t & 1) == 0;
      below[t] = u ? lower_bound_dev<int32_t>(rowdeg, n_u, lim.d[t >> 1])
                   : lower_bound_dev<int32_t>(rowdeg + n_u, n - n_u, lim.d[t >> 1]);
    }
    for (int32_t c = t; c < un.n_graphs; c += blockDim.x) {
      if (un.uo(c + 1) > un.uo(c)) atomicMax(&max_deg[0], (unsigned)rowdeg[un.uo(c + 1) - 1]);
      if (un.vo(c + 1) > un.vo(c)) atomicMax(&max_deg[1], (unsigned)rowdeg[n_u + un.vo(c + 1) - 1]);
    }
    return;
  }
  const int64_t stride = (int64_t)(gridDim.x - 1) * blockDim.x;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride) {
    const int32_t d = rowdeg[r];
    int64_t t;  // side rank threshold in the other side
    if (r < n_u) {
      const int32_t c = un.comp_u(r);
      const int64_t b = un.vo(c), e = un.vo(c + 1);
      t = b + lower_bound_dev<int32_t>(rowdeg + n_u + b, e - b, d);
    } else {
      const int32_t c = un.comp_v(r - n_u);
      const int64_t b = un.uo(c), e = un.uo(c + 1);
      t = b + upper_bound_dev<int32_t>(rowdeg + b, e - b, d);
    }
    const int64_t b = row_ptr[r], e = row_ptr[r + 1];
    lower[r] = (uint32_t)lower_bound_dev<uint32_t>(col + b, e - b, (uint32_t)(t << 1));
    const uint32_t from = (uint32_t)(lone[r < n_u ? 1 : 0] << 1);  // the other side's first rank of degree 2
    int64_t skip = 0;
    if (from && b < e && col[b] < from) skip = lower_bound_dev<uint32_t>(col + b, e - b, from);
    span[r] = make_uint2((uint32_t)(b + skip), (uint32_t)e);
  }
}

// work[p] = sum over lower neighbours v of p of |{w in row(v) : rank(w) < rank(p)}|,
// i.e. the wedges Algorithm 1 accepts at pivot p. Every edge appears as the
// entry at V position m + k (row v, index idx_v in it) and at U position
// upos[k] (row u, index idx_u); rows ascend by rank, so idx_v entries of
// row(v) rank below u and idx_u entries of row(u) rank below v. A lower
// neighbour v of u (idx_u < lower[u]) thus adds idx_v to work[u], and a lower
// neighbour u of v (idx_v < lower[v]) adds idx_u to work[v]. Edges are taken
// in V order, 32 consecutive ones per warp: the V rows' sums are merged by a
// segmented warp sum, the U rows' go to their rows directly.
__global__ void work_kernel(CsrKeys ck, const int64_t* __restrict__ row_ptr, const uint32_t* __restrict__ lower,
                            unsigned long long* __restrict__ work, const unsigned* flags) {
  constexpr int kRound = 4;  // edges per thread per round, their loads in flight together
  if (cta_stopped(flags)) return;
  const int64_t m = ck.m;
  const uint64_t mask_u = (1ull << ck.bits_u) - 1;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t iters = (m + stride - 1) / stride;  // the same for every lane: the warp shuffles together
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const unsigned lane = lane_id();
  for (int64_t it = 0; it < iters; it += kRound) {
    uint64_t key[kRound];
    uint32_t up[kRound];
#pragma unroll
    for (int j = 0; j < kRound; j++) {
      const int64_t k = (it + j) * stride + t0;
      key[j] = k < m ? ck.kv[k] : 0;
      up[j] = k < m ? ck.upos[k] : 0;
    }
    int64_t v[kRound], ru[kRound];
    uint64_t idx_v[kRound], idx_u[kRound];
    uint32_t low_u[kRound], low_v[kRound];
#pragma unroll
    for (int j = 0; j < kRound; j++) {
      const int64_t k = (it + j) * stride + t0;
      ru[j] = (int64_t)((key[j] >> 1) & mask_u);
      v[j] = -1;
      idx_v[j] = idx_u[j] = 0;
      low_u[j] = low_v[j] = 0;
      if (k < m) {
        v[j] = (int64_t)ck.n_u + (int64_t)(key[j] >> (ck.bits_u + 1));
        idx_v[j] = (uint64_t)(m + k - row_ptr[v[j]]);
        idx_u[j] = (uint64_t)((int64_t)up[j] - row_ptr[ru[j]]);
        low_u[j] = lower[ru[j]];
        low_v[j] = lower[v[j]];
      }
    }
#pragma unroll
    for (int j = 0; j < kRound; j++) {
      if (v[j] >= 0 && idx_u[j] < low_u[j] && idx_v[j]) atomicAdd(&work[ru[j]], (unsigned long long)idx_v[j]);
      uint64_t acc = (v[j] >= 0 && idx_v[j] < low_v[j]) ? idx_u[j] : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_down_sync(kFullMask, acc, o);
        const int64_t v2 = __shfl_down_sync(kFullMask, v[j], o);
        if (lane + o < 32 && v2 == v[j]) acc += y;
      }
      const int64_t vp = __shfl_up_sync(kFullMask, v[j], 1);
      if (v[j] >= 0 && acc && (lane == 0 || vp != v[j])) atomicAdd(&work[v[j]], (unsigned long long)acc);
    }
  }
}

struct PrepStats {
  unsigned long long wedges, wedges_hub, wedges_medium, wedges_light;
  unsigned long long n_piv, n_hub, n_medium;
  unsigned long long lower_hub, lower_medium, lower_light;
  unsigned long long max_work;
};
constexpr int kStatSums = 10;  // the sums of PrepStats, in order; max_work follows

// Sums over the hub plan.
struct HubStats {
  unsigned long long items, cursor_inits, cursor_steps, max_lower, list_cap;
};

// What a build reads back from the device.
struct PrepResult {
  PrepStats st;
  HubStats hubs;
  int64_t below[8];         // vertices of degree below four limits (lower_kernel)
  int64_t lone[2];          // a plain graph's vertices of degree 0 and 1 (ranks_kernel)
  unsigned max_deg[2];      // largest degree of each side (lower_kernel)
  unsigned long long kept;  // distinct edges (dedup_kernel)
  unsigned flags;           // kPrep*
};

// Pivots that can close a butterfly: at least two lower neighbours and at
// least one accepted wedge. (A pivot with a single lower neighbour v reaches
// every endpoint w at most once, so all its buckets stay below 2.) One pass
// over tiles of kPivotTile rows adds up the statistics, compacts the pivots in
// row order as sort keys ~work (ascending keys are descending work) with their
// rows, and counts the digits of that sort.
constexpr int kPivotItems = 8;
constexpr int kPivotTile = kRowThreads * kPivotItems;

__global__ void __launch_bounds__(kRowThreads) pivots_kernel(const uint64_t* __restrict__ work,
                                                             const uint32_t* __restrict__ lower, int64_t n,
                                                             uint64_t light_max, uint64_t medium_max,
                                                             uint64_t* __restrict__ key, uint32_t* __restrict__ row,
                                                             uint32_t* hist, PrepStats* st, uint64_t* state,
                                                             unsigned* counter, unsigned* flags) {
  __shared__ uint32_t h[kRsMaxPasses][256];
  __shared__ uint64_t part[kRowThreads / 32][kStatSums + 1];
  __shared__ uint32_t tot_sh;
  const int64_t tile = take_tile(counter, flags);
  if (tile < 0) return;
  DigitCounts dc{h, kRsMaxPasses, 0};
  dc.start();
  const int64_t r0 = tile * kPivotTile + (int64_t)threadIdx.x * kPivotItems;
  uint64_t w[kPivotItems];
  uint64_t s[kStatSums] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  uint64_t mx = 0;
  uint32_t mine = 0;
#pragma unroll
  for (int j = 0; j < kPivotItems; j++) {
    const int64_t r = r0 + j;
    w[j] = r < n ? work[r] : 0;
    const uint32_t L = r < n ? lower[r] : 0u;
    s[0] += w[j];
    if (L >= 2 && w[j] > 0) {
      mine |= 1u << j;
      s[4]++;
      mx = w[j] > mx ? w[j] : mx;
      const int tier = w[j] > medium_max ? 0 : w[j] > light_max ? 1 : 2;  // hub, medium, light
      s[1] += tier == 0 ? w[j] : 0;
      s[2] += tier == 1 ? w[j] : 0;
      s[3] += tier == 2 ? w[j] : 0;
      s[5] += tier == 0;
      s[6] += tier == 1;
      s[7] += tier == 0 ? L : 0;
      s[8] += tier == 1 ? L : 0;
      s[9] += tier == 2 ? L : 0;
    }
  }
#pragma unroll
  for (int k = 0; k < kStatSums; k++) {
    const uint64_t t = warp_sum_u64(s[k]);
    if (lane_id() == 0) part[threadIdx.x >> 5][k] = t;
  }
  mx = warp_max_u64(mx);
  if (lane_id() == 0) part[threadIdx.x >> 5][kStatSums] = mx;
  const uint32_t ex = block_excl_scan<uint32_t, kRowThreads>(__popc(mine), &tot_sh);
  __syncthreads();
  if (threadIdx.x <= kStatSums) {
    unsigned long long* out = reinterpret_cast<unsigned long long*>(st) + threadIdx.x;
    uint64_t t = 0;
    for (int k = 0; k < kRowThreads / 32; k++) {
      const uint64_t x = part[k][threadIdx.x];
      t = threadIdx.x < kStatSums ? t + x : x > t ? x : t;
    }
    if (t && threadIdx.x < kStatSums) atomicAdd(out, (unsigned long long)t);
    if (t && threadIdx.x == kStatSums) atomicMax(out, (unsigned long long)t);
  }
  uint64_t prefix;
  if (!tile_prefix(state, tile, tot_sh, flags, &prefix)) return;
  uint64_t at = prefix + ex;
#pragma unroll
  for (int j = 0; j < kPivotItems; j++) {
    if (mine >> j & 1u) {
      if (DBBC_CHECK(at < (uint64_t)n)) {
        key[at] = ~w[j];
        row[at] = (uint32_t)(r0 + j);
      }
      dc.add(~w[j]);
      at++;
    }
  }
  dc.finish(hist);
}

// Union of several graphs: graph i's local ids are shifted by the sizes of the
// graphs before it; an id out of its own graph's range becomes -1, which the
// build's validation finds. Threads take edges grid-wide (one search for the
// warp's first edge, then a walk over the components its lanes span), so a
// large graph is not left to one CTA: 200 graphs of 6.3M edges in all took
// 414 us with a CTA per graph.
__global__ void union_ids_kernel(const int32_t* __restrict__ u, const int32_t* __restrict__ v,
                                 const int8_t* __restrict__ s, const int64_t* __restrict__ eoff,
                                 const int64_t* __restrict__ uoff, const int64_t* __restrict__ voff, int32_t n_graphs,
                                 int64_t m, int32_t* __restrict__ ou, int32_t* __restrict__ ov,
                                 int8_t* __restrict__ os) {
  let_next_start();
  wait_for_previous();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
    int32_t c = component_of(eoff, n_graphs, i - (int64_t)lane_id());
    while (i >= eoff[c + 1]) c++;
    const int64_t u0 = uoff[c], v0 = voff[c];
    const int32_t x = u[i], y = v[i];
    ou[i] = x >= 0 && x < uoff[c + 1] - u0 ? (int32_t)(u0 + x) : -1;
    ov[i] = y >= 0 && y < voff[c + 1] - v0 ? (int32_t)(v0 + y) : -1;
    os[i] = s[i];
  }
}

// The hub plan: every hub's accepted ranks [0, sp) are split into items of
// roughly equal work. One thread plans one hub; the items are written in hub
// order at positions from a prefix sum over tiles of kRowThreads hubs, each
// with the digit that sorts the list by estimated work. On the host this took
// 0.54 ms of a 20M-edge build (14,682 hubs; the build 3.02 -> 2.53 ms) and 2.0
// ms of a union of 200 small graphs (36,000; 3.42 -> 1.54 ms).
struct HubPlanner {
  const int32_t* order;
  const uint32_t* lower;
  const uint64_t* work;
  const int64_t* below;  // vertices of degree below 2^16, 2^8, 2^4 and 2 (U, V each)
  int64_t n_hub;
  int32_t n_u;
  UnionView un;
  Tuning tune;
  uint32_t window16;  // 16-bit counters of a window
};

// 32-bit counters for a whole hub need this many wedges per counter.
constexpr uint64_t kWideWedgesPerRank = 1;

struct HubPlan {
  SweepItem it;              // row and counter widths; lo, hi and est per item
  uint64_t first, sp, W;
  uint64_t rq, rt, rn, windows;  // quarter, tiny and narrow windows, all windows
  uint64_t spans;
  uint32_t L, window16;
  uint64_t span_windows;     // list mode: windows whose lists fit the scratch
};

// The first rank of window w of the hub (windows numbered in rank order over
// the quarter, tiny, narrow and wide parts).
__device__ __forceinline__ uint64_t window_start(const HubPlan& p, uint64_t w) {
  const uint64_t w16 = p.window16;
  if (w < p.rq) return p.first + w * 4 * w16;
  if (w < p.rq + p.rt) return p.it.q_end + (w - p.rq) * 2 * w16;
  if (w < p.rq + p.rt + p.rn) return p.it.t_end + (w - p.rq - p.rt) * w16;
  return min(p.sp, (uint64_t)p.it.n_end + (w - p.rq - p.rt - p.rn) * (w16 / 2));
}

__device__ __forceinline__ HubPlan plan_hub(const HubPlanner& hp, int64_t i) {
  HubPlan p;
  const int32_t row = hp.order[i];
  const uint32_t L = hp.lower[row];
  const uint64_t W = hp.work[row];
  const bool is_u = row < hp.n_u;
  const uint64_t sp = is_u ? (uint64_t)row : (uint64_t)(row - hp.n_u);
  // the hub's accepted endpoints are the ranks of its own component below it
  const uint64_t start = (uint64_t)(is_u ? hp.un.uo(hp.un.comp_u((int64_t)sp)) : hp.un.vo(hp.un.comp_v((int64_t)sp)));
  // counter widths by the counts they must hold: a count never exceeds the
  // endpoint's degree nor the hub's lower-neighbour count L. Ranks ascend by
  // degree, so quarter (4-bit halves) counters serve the ranks below the
  // side's first endpoint of degree >= 2^4, tiny (8-bit) ones those below
  // degree 2^8 and narrow (16-bit) ones those below degree 2^16; for a union,
  // whose ranks are component-major, only L bounds the counts. Endpoints of
  // degree 0 and 1 (the lowest ranks) are in no span, so the windows start
  // after them: a fifth of the 20M U vertices of the 300M-edge polarized
  // graph, whose sweep that took from 515 to 496 ms. A hub whose endpoints all fit one window of wider counters takes
  // that instead of a window per width: fewer (neighbour, window) visits and
  // barriers, and a 32-bit half that is a word of its own is the cheapest to
  // count in (the class of a wedge picks the word and the increment is 1), if
  // enough wedges share the clearing of its words. Hub sweeps of a 1M-edge
  // graph 0.222 -> 0.197 ms and of a 1.7M-edge one 0.383 -> 0.299 ms; 1,024
  // batched small graphs 3.46 -> 3.14 ms (3.20 without the 32-bit form; one,
  // two or eight wedges per rank make no difference beyond 2%).
  const bool plain = hp.un.n_graphs == 1;
  const int64_t* below = hp.below + (is_u ? 0 : 1);
  auto clamp_rank = [&](int64_t x) { return max(start, min(sp, (uint64_t)max(x, (int64_t)0))); };
  const uint64_t first = plain ? clamp_rank(below[6]) : start;
  uint64_t quarter_end = L < (uint32_t)kQuarterCountLimit ? sp : plain ? max(first, clamp_rank(below[4])) : first;
  uint64_t tiny_end = L < (uint32_t)kTinyCountLimit ? sp : plain ? max(quarter_end,
                                                                       clamp_rank(below[2])) : quarter_end;
  uint64_t narrow_end = L < (uint32_t)kNarrowCountLimit ? sp : plain ? max(tiny_end, clamp_rank(below[0])) : tiny_end;
  const uint64_t full = hp.window16, H4 = 4 * full, H8 = 2 * full;
  const double fin = (double)hp.tune.finalize_window_wedges;
  {  // wider counters where they fit one window
    const uint64_t ranks = sp - first;
    uint64_t words = max(min(quarter_end - first, H4) >> 2, min(tiny_end - quarter_end, H8) >> 1);
    words = max(words, max(min(narrow_end - tiny_end, full), 2 * min(sp - narrow_end, full / 2)));
    // (a narrow CTA's item keeps fitting one)
    const uint64_t limit = W <= kNarrowItemWork && words + 1 <= kNarrowWords ? (uint64_t)kNarrowWords : full;
    const int widths = (quarter_end > first) + (tiny_end > quarter_end) + (narrow_end > tiny_end) + (sp > narrow_end);
    if (2 * ranks <= limit && W >= kWideWedgesPerRank * ranks && (double)W >= fin) {
      quarter_end = tiny_end = narrow_end = first;
    } else if (widths > 1 && ranks <= limit && narrow_end == sp) {
      quarter_end = tiny_end = first;
    }
  }
  p.rq = (quarter_end - first + H4 - 1) / H4;
  p.rt = (tiny_end - quarter_end + H8 - 1) / H8;
  p.rn = (narrow_end - tiny_end + full - 1) / full;
  const uint64_t rw = (sp - narrow_end + full / 2 - 1) / (full / 2);
  p.window16 = hp.window16;
  p.windows = p.rq + p.rt + p.rn + rw;
  p.first = first;
  p.sp = sp;
  p.W = W;
  p.L = L;
  // an item that does not start at the first rank pays one binary search per
  // lower neighbour, so items stay large against the lower-neighbour count
  const uint64_t target = max(hp.tune.hub_item_work, (uint64_t)64 * L);
  // lanes per (neighbour, window) segment from the hub's mean segment length
  const double density = (double)W / ((double)L * (double)max((uint64_t)1, p.windows));
  const double* gd = hp.tune.group_density;
  const int dense_log = density >= gd[0] ? 5 : density >= gd[1] ? 4 : density >= gd[2] ? 3 : density >= gd[3] ? 2 : 0;
  // sparse hubs sweep in list mode: one item per hub, run in spans of at most
  // span_windows windows whose lists (plus two overflow lists of L slots) fit
  // the per-CTA list scratch
  const uint64_t per_nb = (uint64_t)kListCapEntries / max(L, 1u);
  p.span_windows = per_nb >= 3 ? min((uint64_t)kListMaxWindows, per_nb - 2) : 0;
  const bool listed = density < hp.tune.list_density && p.span_windows >= 1 && p.windows >= 2;
  // list-mode items take list_group_log lanes per segment, at least 8 when
  // their mean segment reaches list_wide_density
  const int list_log =
      density >= hp.tune.list_wide_density ? max(3, hp.tune.list_group_log) : hp.tune.list_group_log;
  // items of roughly `target` wedges over consecutive windows (one item in
  // list mode); an item crosses width boundaries freely
  p.spans = p.windows == 0 ? 0 : listed ? 1 : max((uint64_t)1, min(p.windows, W / target));
  p.it.row = row;
  p.it.q_end = (uint32_t)quarter_end;
  p.it.t_end = (uint32_t)tiny_end;
  p.it.n_end = (uint32_t)narrow_end;
  p.it.group_log = (int16_t)(listed ? list_log : dense_log);
  p.it.flags = listed ? kItemList : 0;
  // dense items: finalise each window from its counters when clearing it
  if (p.windows && (double)W / (double)p.windows >= fin)
    p.it.flags |= kItemFinalize;
  p.it.est = p.spans ? (uint32_t)min((uint64_t)0xFFFFFFFFu, max((uint64_t)1, W / p.spans)) : 0u;
  return p;
}

__global__ void __launch_bounds__(kRowThreads) plan_hubs_kernel(HubPlanner hp, SweepItem* __restrict__ items,
                                                                uint64_t cap, uint64_t* __restrict__ key,
                                                                uint32_t* __restrict__ idx, uint32_t* hist,
                                                                HubStats* st, uint64_t* state, unsigned* counter,
                                                                unsigned* flags) {
  __shared__ uint32_t h[1][256];
  __shared__ uint64_t tot_sh;
  const int64_t tile = take_tile(counter, flags);
  if (tile < 0) return;
  DigitCounts dc{h, 1, 0};
  dc.start();
  const int64_t i = tile * kRowThreads + threadIdx.x;
  HubPlan p{};
  if (i < hp.n_hub) p = plan_hub(hp, i);
  const uint64_t ex = block_excl_scan<uint64_t, kRowThreads>(p.spans, &tot_sh);
  __syncthreads();
  uint64_t prefix;
  if (!tile_prefix(state, tile, tot_sh, flags, &prefix)) return;
  if (threadIdx.x == 0) atomicAdd(&st->items, (unsigned long long)tot_sh);
  const bool listed = (p.it.flags & kItemList) != 0;
  for (uint64_t k = 0; k < p.spans; k++) {
    const uint64_t w0 = p.windows * k / p.spans, w1 = p.windows * (k + 1) / p.spans;
    SweepItem it = p.it;
    it.lo = (uint32_t)window_start(p, w0);
    it.hi = (uint32_t)(w1 == p.windows ? p.sp : window_start(p, w1));
    if (w0 == 0) it.flags |= kItemFirst;
    const uint64_t at = prefix + ex + k;
    if (at >= cap) {  // cannot happen: cap bounds the number of items
      (void)DBBC_CHECK(false);
      break;
    }
    items[at] = it;
    idx[at] = (uint32_t)at;
    const uint64_t d = estimate_digit(it.est, 3, 256u);
    key[at] = d;
    dc.add(d);
  }
  const uint64_t inits = warp_sum_u64(p.spans * p.L), steps = warp_sum_u64(listed ? 0 : p.windows * p.L);
  const uint64_t low = warp_max_u64(p.spans ? p.L : 0);
  const uint64_t slots = warp_max_u64(listed ? (min(p.windows, p.span_windows) + 2) * p.L : 0);
  if (lane_id() == 0 && inits) {
    atomicAdd(&st->cursor_inits, (unsigned long long)inits);
    atomicMax(&st->max_lower, (unsigned long long)low);
    if (steps) atomicAdd(&st->cursor_steps, (unsigned long long)steps);
    if (slots) atomicMax(&st->list_cap, (unsigned long long)slots);
  }
  dc.finish(hist);
}

// ------------------------------------------------------------------ host
static unsigned grid_for(int64_t n, int threads = 256) {
  int64_t b = ceil_div<int64_t>(n > 0 ? n : 1, threads);
  const int64_t cap = (int64_t)kNumSMs * 16;
  return (unsigned)(b < cap ? b : cap);
}

// For kernels that count digits: one resident wave, so that few CTAs add to
// the global counts.
static unsigned count_grid(int64_t n) { return std::min(grid_for(n), (unsigned)kNumSMs * 8u); }

void* graph_alloc(dbbc_graph* g, size_t bytes, size_t pad) {
  void* p = dev_alloc((bytes ? bytes : 16) + pad, g->stream);
  if (!p) throw Error{DBBC_ENOMEM, "graph_alloc"};
  g->allocations.push_back(p);
  g->device_bytes += bytes;
  return p;
}

// Give one of the graph's allocations back.
static void graph_release(dbbc_graph* g, void* p, size_t bytes) {
  g->allocations.erase(std::find(g->allocations.begin(), g->allocations.end(), p));
  g->device_bytes -= bytes;
  dev_free(p, g->stream);
}

void free_graph_memory(dbbc_graph* g) {
  for (void* p : g->allocations) dev_free(p, g->stream);
  g->allocations.clear();
  g->device_bytes = 0;
}

template <typename T>
static T read_back(const T* d, cudaStream_t s) {
  T h;
  DBBC_CUDA(cudaMemcpyAsync(&h, d, sizeof(T), cudaMemcpyDeviceToHost, s));
  DBBC_CUDA(cudaStreamSynchronize(s));
  return h;
}

// Carves a build's device scratch out of one allocation: run once without a
// base to size it, then again to place it.
struct Carver {
  char* base = nullptr;
  size_t used = 0;
  template <typename T>
  T* get(size_t n) {
    T* p = reinterpret_cast<T*>(base + used);
    used += (n * sizeof(T) + 255) / 256 * 256;
    return p;
  }
  RadixState radix(int passes, int64_t n) {
    RadixState r;
    r.hist = get<uint32_t>((size_t)passes * 256);
    r.counters = get<unsigned>((size_t)passes);
    r.state = get<uint32_t>((size_t)passes * (size_t)radix_tiles(n) * 256);
    return r;
  }
};

// Plans the hubs on the device, behind the pivot sort; returns once the
// items are counted. Throws when a bounded wait of the build gave up.
static void plan_hubs(dbbc_graph* g, cudaStream_t s, const UnionView& un, PrepResult* res, uint64_t max_work,
                      Scratch& sc) {
  if (g->n_hub == 0) return;
  // Two half CTAs per SM hide each other's barriers and window ends, at the
  // price of up to twice the windows. They pay where the sides are small and no
  // hub alone would keep a half CTA busy past the others' end: hub sweeps of a
  // 1M-edge graph 0.198 -> 0.167 ms and of a 1.7M-edge one 0.301 -> 0.241 ms;
  // where one large hub outlasts the rest (151k edges) 0.101 -> 0.129 ms, with
  // larger sides (9.2M edges, 540k vertices) 3.8 -> 4.8 ms. The plan's windows,
  // and with them its lanes per segment, are the half CTAs' although plans,
  // unions and the per-vertex and per-edge sweeps run its items with windows of
  // their own: against a plan for full windows these took between 3% less and
  // 7% more time (ratings graphs of 1M, 2M and 4M edges).
  const int64_t half_ctas = 2 * (int64_t)num_sms();
  g->half_ctas = std::max(g->n_u, g->n_v) <= kHalfMaxSide &&
                 max_work <= 4 * (g->wedges_hub / (uint64_t)half_ctas);
  // a hub has at most W / hub_item_work items, rounded up, and no more than windows
  const uint64_t side = (uint64_t)std::max(g->n_u, g->n_v);
  const uint32_t window16 = g->half_ctas ? kHalfWindow16 : kSweepWindow16;
  const uint64_t cap = std::min((uint64_t)g->n_hub + g->wedges_hub / g->tune.hub_item_work,
                                (uint64_t)g->n_hub * (side / (window16 / 2) + 4));
  const int64_t tiles = ceil_div<int64_t>(g->n_hub, kRowThreads);
  struct Layout {
    RadixState sort;
    uint64_t* state;
    unsigned* counter;
    size_t zeroed;
    SweepItem* items;
    uint64_t* key;
    uint32_t *idx, *sorted;
  };
  auto place = [&](Carver& c) {
    Layout l;
    l.sort = c.radix(1, (int64_t)cap);
    l.state = c.get<uint64_t>((size_t)tiles);
    l.counter = c.get<unsigned>(1);
    l.zeroed = c.used;
    l.items = c.get<SweepItem>(cap);
    l.key = c.get<uint64_t>(cap);
    l.idx = c.get<uint32_t>(cap);
    l.sorted = c.get<uint32_t>(cap);
    return l;
  };
  Carver carver;
  place(carver);
  carver.base = sc.get<char>(carver.used);
  char* const zero = carver.base;
  carver.used = 0;
  const Layout l = place(carver);
  DBBC_CUDA(cudaMemsetAsync(zero, 0, l.zeroed, s));
  const HubPlanner hp{g->order, g->lower, g->work, res->below, g->n_hub, g->n_u, un, g->tune, window16};
  launch_overlapped(plan_hubs_kernel,
                    (unsigned)tiles, kRowThreads, 0, s, hp, l.items, cap, l.key, l.idx, l.sort.hist, &res->hubs,
                    l.state, l.counter, &res->flags);
  const PrepResult r = read_back(res, s);
  if (r.flags & kPrepTimeout) throw Error{DBBC_EINTERNAL, "a bounded wait of the build gave up"};
  if (r.hubs.items > cap) throw Error{DBBC_EINTERNAL, "hub plan"};
  g->n_sweep_items = (int64_t)r.hubs.items;
  g->hub_cursor_inits = (int64_t)r.hubs.cursor_inits;
  g->hub_cursor_steps = (int64_t)r.hubs.cursor_steps;
  g->sweep_max_lower = std::max<int64_t>(1, (int64_t)r.hubs.max_lower);
  g->sweep_list_cap = (int64_t)r.hubs.list_cap;
  g->sweep_items = static_cast<SweepItem*>(graph_alloc(g, (size_t)g->n_sweep_items * sizeof(SweepItem)));
  if (g->n_sweep_items == 0) return;
  radix_pass<PlainLoad, true, false, false>(PlainLoad{l.key, l.idx}, PassOut{nullptr, l.sorted, nullptr, 0},
                                            g->n_sweep_items, 0, 0, l.sort, &res->flags, s);
  launch_overlapped(gather_kernel<SweepItem>, grid_for(g->n_sweep_items), 256, 0, s, l.items, l.sorted,
                    g->n_sweep_items, g->sweep_items, &res->flags);
}

void build_graph_multi(dbbc_graph* g, const int32_t* u, const int32_t* v, const int8_t* sgn,
                       const int64_t* edge_offsets, const int32_t* n_u, const int32_t* n_v, int32_t n_graphs,
                       bool on_device, bool reject_duplicates, cudaStream_t s) {
  // host metadata: edge ranges and the id shift of every graph
  std::vector<int64_t> uoff((size_t)n_graphs + 1, 0), voff((size_t)n_graphs + 1, 0);
  for (int32_t i = 0; i < n_graphs; i++) {
    if (n_u[i] < 0 || n_v[i] < 0 || edge_offsets[i + 1] < edge_offsets[i])
      throw Error{DBBC_EINVAL, "bad component sizes or edge offsets"};
    uoff[(size_t)i + 1] = uoff[(size_t)i] + n_u[i];
    voff[(size_t)i + 1] = voff[(size_t)i] + n_v[i];
  }
  const int64_t m = edge_offsets[n_graphs] - edge_offsets[0];
  if (edge_offsets[0] != 0 || m >= (int64_t{1} << 31) || uoff.back() + voff.back() >= (int64_t{1} << 31))
    throw Error{DBBC_EINVAL, "union too large"};
  g->n_u = (int32_t)uoff.back();
  g->n_v = (int32_t)voff.back();
  Scratch sc(s);
  const int32_t* du = u;
  const int32_t* dv = v;
  const int8_t* ds = sgn;
  if (!on_device && m > 0) {
    int32_t* tu = sc.get<int32_t>((size_t)m);
    int32_t* tv = sc.get<int32_t>((size_t)m);
    int8_t* ts = sc.get<int8_t>((size_t)m);
    DBBC_CUDA(cudaMemcpyAsync(tu, u, (size_t)m * 4, cudaMemcpyHostToDevice, s));
    DBBC_CUDA(cudaMemcpyAsync(tv, v, (size_t)m * 4, cudaMemcpyHostToDevice, s));
    DBBC_CUDA(cudaMemcpyAsync(ts, sgn, (size_t)m, cudaMemcpyHostToDevice, s));
    du = tu;
    dv = tv;
    ds = ts;
  }
  // edge, U and V offsets in one upload
  const size_t k = (size_t)n_graphs + 1;
  std::vector<int64_t> meta(3 * k);
  const WaitOnThrow wait_for_copy{s};
  std::copy(edge_offsets, edge_offsets + k, meta.begin());
  std::copy(uoff.begin(), uoff.end(), meta.begin() + (ptrdiff_t)k);
  std::copy(voff.begin(), voff.end(), meta.begin() + (ptrdiff_t)(2 * k));
  int64_t* d_meta = sc.get<int64_t>(meta.size());
  DBBC_CUDA(cudaMemcpyAsync(d_meta, meta.data(), meta.size() * 8, cudaMemcpyHostToDevice, s));
  int32_t* ou = sc.get<int32_t>((size_t)std::max<int64_t>(m, 1));
  int32_t* ov = sc.get<int32_t>((size_t)std::max<int64_t>(m, 1));
  int8_t* os = sc.get<int8_t>((size_t)std::max<int64_t>(m, 1));
  if (m > 0) {
    launch_overlapped(union_ids_kernel,
                      grid_for(m), 256, 0, s, du, dv, ds, d_meta, d_meta + k, d_meta + 2 * k, n_graphs, m, ou, ov, os);
  }
  UnionSpec un;
  un.n_graphs = std::max<int32_t>(n_graphs, 1);
  un.uoff = n_graphs > 0 ? uoff : std::vector<int64_t>{0, 0};
  un.voff = n_graphs > 0 ? voff : std::vector<int64_t>{0, 0};
  un.d_uoff = d_meta + k;
  un.d_voff = d_meta + 2 * k;
  for (int32_t i = 0; i < n_graphs; i++) un.max_side = std::max<int64_t>(un.max_side, std::max(n_u[i], n_v[i]));
  g->n_components = n_graphs;
  g->component = static_cast<int32_t*>(graph_alloc(g, (size_t)std::max<int64_t>((int64_t)g->n_u + g->n_v, 1) * 4));
  build_graph(g, ou, ov, os, m, true, reject_duplicates, s, &un);
}

void build_graph(dbbc_graph* g, const int32_t* u_in, const int32_t* v_in, const int8_t* s_in, int64_t m,
                 bool on_device, bool reject_duplicates, cudaStream_t s, const UnionSpec* union_spec) {
  const int32_t n_u = g->n_u, n_v = g->n_v;
  const int64_t n = (int64_t)n_u + n_v;
  g->n = n;
  g->m_input = m;
  g->tune = current_tuning();
  // a plain graph is a union of one component
  UnionSpec plain;
  const UnionSpec* un = union_spec;
  if (!un) {
    plain.uoff = {0, (int64_t)n_u};
    plain.voff = {0, (int64_t)n_v};
    plain.max_side = std::max<int64_t>(n_u, n_v);
    un = &plain;
  }
  const UnionView uv{un->d_uoff, un->d_voff, un->n_graphs, n_u, n_v};

  const int bits_u = bits_for(n_u > 0 ? (uint64_t)(n_u - 1) : 0);
  const int bits_v = bits_for(n_v > 0 ? (uint64_t)(n_v - 1) : 0);
  // rank keys: (side, component, degree, id within the component)
  const int bits_comp = un->n_graphs > 1 ? bits_for((uint64_t)(un->n_graphs - 1)) : 0;
  const int bits_lid = std::max(1, bits_for(un->max_side > 0 ? (uint64_t)(un->max_side - 1) : 0));
  const int bits_deg = std::max(1, bits_for((uint64_t)un->max_side));
  if (1 + bits_comp + bits_deg + bits_lid > 64) throw Error{DBBC_EINVAL, "union too large for 64-bit rank keys"};
  // keys are generated in (side, component, local id) order, so a stable sort
  // on (side, component, degree) alone leaves equal degrees by id; the edge
  // sorts skip bit 0 (the sign), so repeated pairs stay in input order
  const int rank_end = 1 + bits_comp + bits_deg + bits_lid;
  const int passes_r = radix_passes(bits_lid, rank_end);
  const int passes_u = radix_passes(1, 1 + bits_v + bits_u);
  const int passes_v = radix_passes(1 + bits_u, 1 + bits_u + bits_v);

  // ---- scratch, one allocation: what has to start at zero comes first
  struct Layout {
    PrepResult* res;
    RadixState rank, su, sv, piv;
    uint64_t *row_state, *pivot_state, *dedup_state;
    unsigned* counters;  // tiles of the row, pivot and dedup kernels
    int32_t* deg;
    size_t zeroed;
    int32_t *side_rank, *rowdeg;
    uint64_t *vk0, *vk1, *ck0, *ck1;  // vertex / pivot keys, edge keys
    uint32_t *up0, *up1, *pr0, *pr1;  // U positions, pivot rows
    int32_t *tu, *tv;                 // host inputs; distinct edges
    int8_t* ts;
  };
  auto place = [&](Carver& c) {
    Layout l;
    const size_t mm = (size_t)m, nn = (size_t)n;
    l.res = c.get<PrepResult>(1);
    l.rank = c.radix(passes_r, n);
    l.su = c.radix(passes_u, m);
    l.sv = c.radix(passes_v, m);
    l.piv = c.radix(kRsMaxPasses, n);
    l.row_state = c.get<uint64_t>((size_t)ceil_div<int64_t>(n, kRowTile) + 1);
    l.pivot_state = c.get<uint64_t>((size_t)ceil_div<int64_t>(n, kPivotTile) + 1);
    l.dedup_state = c.get<uint64_t>((size_t)ceil_div<int64_t>(m, kRowTile) + 1);
    l.counters = c.get<unsigned>(3);
    l.deg = c.get<int32_t>(nn);
    l.zeroed = c.used;
    l.side_rank = c.get<int32_t>(nn);
    l.rowdeg = c.get<int32_t>(nn);
    l.vk0 = c.get<uint64_t>(nn);
    l.vk1 = c.get<uint64_t>(nn);
    l.ck0 = c.get<uint64_t>(mm);
    l.ck1 = c.get<uint64_t>(mm);
    l.up0 = c.get<uint32_t>(mm);
    l.up1 = c.get<uint32_t>(mm);
    l.pr0 = c.get<uint32_t>(nn);
    l.pr1 = c.get<uint32_t>(nn);
    l.tu = l.tv = nullptr;
    l.ts = nullptr;
    if (!on_device) {
      l.tu = c.get<int32_t>(mm);
      l.tv = c.get<int32_t>(mm);
      l.ts = c.get<int8_t>(mm);
    }
    return l;
  };
  Scratch sc(s);
  Carver carver;
  place(carver);
  carver.base = sc.get<char>(carver.used);
  carver.used = 0;
  const Layout l = place(carver);
  unsigned* d_flags = &l.res->flags;

  // ---- inputs on the device
  const int32_t* du = u_in;
  const int32_t* dv = v_in;
  const int8_t* ds = s_in;
  if (!on_device && m > 0) {
    DBBC_CUDA(cudaMemcpyAsync(l.tu, u_in, (size_t)m * 4, cudaMemcpyHostToDevice, s));
    DBBC_CUDA(cudaMemcpyAsync(l.tv, v_in, (size_t)m * 4, cudaMemcpyHostToDevice, s));
    DBBC_CUDA(cudaMemcpyAsync(l.ts, s_in, (size_t)m, cudaMemcpyHostToDevice, s));
    du = l.tu;
    dv = l.tv;
    ds = l.ts;
  }
  g->vertex = static_cast<int32_t*>(graph_alloc(g, (size_t)n * 4));
  g->row_ptr = static_cast<int64_t*>(graph_alloc(g, (size_t)(n + 1) * 8));
  g->lower = static_cast<uint32_t*>(graph_alloc(g, (size_t)n * 4));
  g->work = static_cast<uint64_t*>(graph_alloc(g, (size_t)n * 8));
  g->span = static_cast<uint2*>(graph_alloc(g, (size_t)n * sizeof(uint2)));
  if (n == 0) DBBC_CUDA(cudaMemsetAsync(g->row_ptr, 0, 8, s));

  // a1-a4 for an edge list, without a wait: validation and degrees, Def. 3
  // ranks per side, the CSR of both sides, accepted wedges per pivot and the
  // pivots. When an edge is invalid, a (u, v) pair occurs twice or a wait gave
  // up, the kernels that follow return at once and the flags say why. *ku_out
  // gets the U-sorted keys.
  const uint64_t* ku = nullptr;
  void* col_block = nullptr;  // the allocation that holds g->col
  auto build_from_edges = [&](const int32_t* eu, const int32_t* ev, const int8_t* es, int64_t me) -> PrepResult {
    DBBC_CUDA(cudaMemsetAsync(l.res, 0, l.zeroed, s));
    col_block = graph_alloc(g, (size_t)(2 * me) * 4, kColPad + kColAlign);
    g->col = reinterpret_cast<uint32_t*>(((uintptr_t)col_block + kColAlign - 1) / kColAlign * kColAlign);
    if (me > 0)
      launch_overlapped(degree_kernel, grid_for(me), 256, 0, s, eu, ev, es, me, n_u, n_v, l.deg, d_flags);
    if (n > 0) {
      launch_overlapped(vertex_keys_kernel,
                        count_grid(n), 256, 0, s, l.deg, n, n_u, bits_comp, bits_deg, bits_lid, uv, l.vk0, passes_r,
                        l.rank.hist, d_flags);
      uint64_t *in = l.vk0, *out = l.vk1;
      for (int p = 0; p < passes_r; p++, std::swap(in, out))
        radix_pass<PlainLoad, false, true, false>(PlainLoad{in, nullptr}, PassOut{out, nullptr, nullptr, 0}, n,
                                                  bits_lid, p, l.rank, d_flags, s);
      launch_overlapped(ranks_kernel,
                        (unsigned)ceil_div<int64_t>(n, kRowTile), kRowThreads, 0, s, in, n, n_u, bits_comp, bits_deg,
                        bits_lid, uv, g->vertex, l.side_rank, l.rowdeg, g->row_ptr, g->component, g->work, l.res->lone,
                        l.row_state, l.counters, d_flags);
    }
    CsrKeys ck{nullptr, nullptr, me, n_u, bits_u};
    if (me > 0) {
      launch_overlapped(csr_u_keys_kernel,
                        count_grid(me), 256, 0, s, eu, ev, es, me, n_u, l.side_rank, bits_v, l.ck0, passes_u,
                        l.su.hist, d_flags);
      uint64_t *in = l.ck0, *out = l.ck1;
      for (int p = 0; p < passes_u; p++, std::swap(in, out)) {
        const PassOut po{out, nullptr, g->col, (2ull << bits_v) - 1};
        if (p + 1 < passes_u)
          radix_pass<PlainLoad, false, true, false>(PlainLoad{in, nullptr}, po, me, 1, p, l.su, d_flags, s);
        else
          radix_pass<PlainLoad, false, true, true>(PlainLoad{in, nullptr}, po, me, 1, p, l.su, d_flags, s);
      }
      ku = in;
      const VKey vk{bits_u, bits_v};
      launch_overlapped(csr_v_digits_kernel, count_grid(me), 256, 0, s, ku, me, vk, passes_v, l.sv.hist, d_flags);
      uint32_t *vin = l.up0, *vout = l.up1;
      for (int p = 0; p < passes_v; p++, std::swap(in, out), std::swap(vin, vout)) {
        const PassOut po{out, vout, g->col + me, (2ull << bits_u) - 1};
        const bool last = p + 1 == passes_v;
        const VKeyLoad first{ku, vk};
        const PlainLoad next{in, vin};
        if (p == 0 && last) radix_pass<VKeyLoad, true, true, true>(first, po, me, 1 + bits_u, p, l.sv, d_flags, s);
        else if (p == 0) radix_pass<VKeyLoad, true, true, false>(first, po, me, 1 + bits_u, p, l.sv, d_flags, s);
        else if (last) radix_pass<PlainLoad, true, true, true>(next, po, me, 1 + bits_u, p, l.sv, d_flags, s);
        else radix_pass<PlainLoad, true, true, false>(next, po, me, 1 + bits_u, p, l.sv, d_flags, s);
      }
      ck.kv = in;
      ck.upos = vin;
    }
    if (n > 0) {
      const DegreeLimits lim{{kNarrowCountLimit, kTinyCountLimit, kQuarterCountLimit, 2}};
      launch_overlapped(lower_kernel,
                        grid_for(n) + 1, 256, 0, s, g->row_ptr, g->col, l.rowdeg, n, n_u, uv, g->lower, g->span,
                        l.res->lone, lim,
                        l.res->below, l.res->max_deg, d_flags);
      if (me > 0)
        launch_overlapped(work_kernel, grid_for(me), 256, 0, s, ck, g->row_ptr, g->lower,
                          reinterpret_cast<unsigned long long*>(g->work), d_flags);
      launch_overlapped(pivots_kernel,
                        (unsigned)ceil_div<int64_t>(n, kPivotTile), kRowThreads, 0, s, g->work, g->lower, n,
                        g->tune.light_max_work, g->tune.medium_max_work, l.vk0, l.pr0, l.piv.hist, &l.res->st,
                        l.pivot_state, l.counters + 1, d_flags);
    }
    const PrepResult r = read_back(l.res, s);
    if (r.flags & kPrepInvalid) throw Error{DBBC_EINVAL, "invalid edge id or sign"};
    if (r.flags & kPrepTimeout) throw Error{DBBC_EINTERNAL, "a bounded wait of the build gave up"};
    return r;
  };

  // ---- build straight from the input; only when some (u, v) pair repeats,
  // keep the latest occurrence of every pair (the last of its run in the
  // U-sorted list) and build again from the distinct edges.
  int64_t mu = m;
  PrepResult r = build_from_edges(du, dv, ds, m);
  if (r.flags & kPrepDup) {
    if (reject_duplicates) throw Error{DBBC_EINVAL, "duplicate edge under DBBC_DUP_REJECT"};
    int32_t* eu = sc.get<int32_t>((size_t)m);
    int32_t* ev = sc.get<int32_t>((size_t)m);
    int8_t* es = sc.get<int8_t>((size_t)m);
    DBBC_CUDA(cudaMemsetAsync(d_flags, 0, sizeof(unsigned), s));
    launch_overlapped(dedup_kernel,
                      (unsigned)ceil_div<int64_t>(m, kRowTile), kRowThreads, 0, s, ku, m, bits_v, n_u, n, g->vertex,
                      eu, ev, es, reinterpret_cast<uint64_t*>(&l.res->kept), l.dedup_state, l.counters + 2, d_flags);
    const PrepResult d = read_back(l.res, s);
    if (d.flags & kPrepTimeout) throw Error{DBBC_EINTERNAL, "a bounded wait of the build gave up"};
    mu = (int64_t)d.kept;
    graph_release(g, col_block, (size_t)(2 * m) * 4);
    g->col = nullptr;
    r = build_from_edges(eu, ev, es, mu);
    if (r.flags & kPrepDup) throw Error{DBBC_EINTERNAL, "duplicates left after deduplication"};
  }
  g->m = mu;
  g->nnz = 2 * mu;

  // ---- the counting tiers: pivots in descending work, ties by row
  const PrepStats& st = r.st;
  g->wedges = st.wedges;
  g->wedges_hub = st.wedges_hub;
  g->wedges_medium = st.wedges_medium;
  g->wedges_light = st.wedges_light;
  g->n_piv = (int64_t)st.n_piv;
  g->n_hub = (int64_t)st.n_hub;
  g->n_medium = (int64_t)st.n_medium;
  g->n_light = g->n_piv - g->n_hub - g->n_medium;
  g->lower_hub = (int64_t)st.lower_hub;
  g->lower_medium = (int64_t)st.lower_medium;
  g->lower_light = (int64_t)st.lower_light;
  g->order = static_cast<int32_t*>(graph_alloc(g, (size_t)std::max<int64_t>(g->n_piv, 1) * 4));
  if (g->n_piv > 0) {
    const int passes = radix_passes(0, bits_for(st.max_work));
    uint64_t *kin = l.vk0, *kout = l.vk1;
    uint32_t *vin = l.pr0, *vout = l.pr1;
    for (int p = 0; p < passes; p++, std::swap(kin, kout), std::swap(vin, vout)) {
      const PlainLoad in{kin, vin};
      if (p + 1 == passes)
        radix_pass<PlainLoad, true, false, false>(
            in, PassOut{nullptr, reinterpret_cast<uint32_t*>(g->order), nullptr, 0}, g->n_piv, 0, p, l.piv, d_flags,
            s);
      else
        radix_pass<PlainLoad, true, true, false>(in, PassOut{kout, vout, nullptr, 0}, g->n_piv, 0, p, l.piv, d_flags,
                                                 s);
    }
  }
  g->max_deg_u = r.max_deg[0];
  g->max_deg_v = r.max_deg[1];
  plan_hubs(g, s, uv, l.res, st.max_work, sc);
  if (read_back(d_flags, s) & kPrepTimeout) throw Error{DBBC_EINTERNAL, "a bounded wait of the build gave up"};
}

}  // namespace dbbc
