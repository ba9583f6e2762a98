// In-repo device primitives: single-pass prefix sums over tiles and a stable
// LSD radix sort with one kernel per digit. Written for sm_103a; no CUB.
//
// Both chain their tiles by decoupled look-back (Merrill and Garland,
// "Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016; one kernel
// per radix digit that way: Adinets and Merrill, "Onesweep: A Faster Least
// Significant Digit Radix Sort for GPUs", 2022): a tile
// publishes its own sum, adds up what the tiles before it have published until
// it meets one whose running total is known, and publishes its own running
// total. Tiles are numbered by a counter in the order in which their CTAs
// start, so every tile that one waits for is running or done. Each wait is
// bounded all the same: a tile that polls kSpinLimit times sets kPrepTimeout in
// the pass's flag word and returns, every other wait then ends at once, and
// the kernels that follow (gather_kernel included: its indexes are then partly
// unwritten) see the flag and return.
#pragma once

#include <algorithm>

#include "common.cuh"

namespace dbbc {

// Bits of a build's device flag word. kPrepStop: the kernels after the one
// that set it have nothing valid to work on and return.
enum : unsigned {
  kPrepBadU = 1u,
  kPrepBadV = 2u,
  kPrepBadSign = 4u,
  kPrepInvalid = kPrepBadU | kPrepBadV | kPrepBadSign,
  kPrepDup = 8u,       // a (u, v) pair occurs twice
  kPrepTimeout = 16u,  // a bounded wait gave up
  kPrepStop = kPrepInvalid | kPrepDup | kPrepTimeout,
};

// Polls of one wait (seconds; a wait normally takes microseconds). With 0, for
// tests of what follows a wait that gave up, every tile but a pass's first one
// gives up before it polls.
#ifndef DBBC_SPIN_LIMIT
#define DBBC_SPIN_LIMIT (1u << 22)
#endif
constexpr uint32_t kSpinLimit = DBBC_SPIN_LIMIT;

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// True when a wait that has polled `polls` times has to end: it reached its
// limit (which sets the flag), or another one did.
__device__ __forceinline__ bool wait_over(uint32_t polls, unsigned* flags) {
  if (polls >= kSpinLimit) {
    atomicOr(flags, (unsigned)kPrepTimeout);
    return true;
  }
  return (polls & 63u) == 63u && (ld_relaxed(flags) & kPrepTimeout) != 0;
}

// Whether a tile may wait for the ones before it (always, but for kSpinLimit 0).
__device__ __forceinline__ bool may_wait(int64_t tile, unsigned* flags) {
  if (kSpinLimit > 0 || tile == 0) return true;
  atomicOr(flags, (unsigned)kPrepTimeout);
  return false;
}

// ------------------------------------------------------------------ scans
// Inclusive warp scan.
template <typename T>
__device__ __forceinline__ T warp_incl_scan(T x) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(kFullMask, x, o);
    if ((int)lane_id() >= o) x += y;
  }
  return x;
}

// Exclusive block scan of one value per thread (blockDim.x == THREADS, a
// multiple of 32, at most 1024). Returns the exclusive prefix; *total gets the
// block sum. Contains __syncthreads.
template <typename T, int THREADS>
__device__ __forceinline__ T block_excl_scan(T x, T* total) {
  __shared__ T warp_tot[THREADS / 32];
  const int w = threadIdx.x >> 5;
  T inc = warp_incl_scan(x);
  if (lane_id() == 31) warp_tot[w] = inc;
  __syncthreads();
  if (w == 0) {
    T t = lane_id() < THREADS / 32 ? warp_tot[lane_id()] : T(0);
    T ti = warp_incl_scan(t);
    if (lane_id() < THREADS / 32) warp_tot[lane_id()] = ti - t;
    if (lane_id() == THREADS / 32 - 1) *total = ti;  // caller's shared slot
  }
  __syncthreads();
  return warp_tot[w] + inc - x;
}

// Called first by the build's kernels (see launch_overlapped): whether this CTA
// has to return at once (kPrepStop), the same answer in every thread although
// other CTAs may be setting the flag. Contains __syncthreads.
__device__ __forceinline__ bool cta_stopped(const unsigned* flags) {
  let_next_start();
  wait_for_previous();
  return __syncthreads_or(threadIdx.x == 0 && (ld_relaxed(flags) & kPrepStop) != 0) != 0;
}

// The same for kernels over tiles: the number of this CTA's tile, or -1 when
// the CTA has to return. Contains __syncthreads.
__device__ __forceinline__ int64_t take_tile(unsigned* counter, const unsigned* flags) {
  let_next_start();
  wait_for_previous();
  __shared__ int64_t tile_sh;
  if (threadIdx.x == 0) {
    const unsigned t = atomicAdd(counter, 1u);  // both requests in flight together
    tile_sh = (ld_relaxed(flags) & kPrepStop) != 0 ? -1 : (int64_t)t;
  }
  __syncthreads();
  return tile_sh;
}

// Exclusive prefix of `sum` over the tiles before this one (sums below 2^62).
// Called by all threads; `state` (one zeroed word per tile) holds 0 (nothing
// yet), kTileSum | sum or kTileTotal | running total. Warp 0 looks at 32
// earlier tiles at a time. Returns false when a wait gave up.
constexpr uint64_t kTileSum = 1ull << 62, kTileTotal = 2ull << 62, kTileValue = kTileSum - 1;

__device__ __forceinline__ bool tile_prefix(uint64_t* state, int64_t tile, uint64_t sum, unsigned* flags,
                                            uint64_t* prefix) {
  __shared__ uint64_t pre_sh;
  __shared__ int ok_sh;
  if (threadIdx.x < 32) {
    const unsigned lane = lane_id();
    if (lane == 0) st_relaxed(&state[tile], (tile == 0 ? kTileTotal : kTileSum) | sum);
    uint64_t pre = 0;
    bool ok = may_wait(tile, flags);
    int64_t end = tile;  // the tiles [end, tile) are in `pre`
    uint32_t polls = 0;
    while (ok && end > 0) {
      const int64_t t = end - 1 - (int64_t)lane;
      const uint64_t s = t >= 0 ? ld_relaxed(&state[t]) : kTileTotal;
      // lanes up to the first running total count, if all before it are there
      const unsigned total = __ballot_sync(kFullMask, (s & kTileTotal) != 0);
      const unsigned none = __ballot_sync(kFullMask, (s & (kTileTotal | kTileSum)) == 0);
      const unsigned upto = total ? (total & (0u - total)) : 0u;            // its bit
      const unsigned need = total ? (upto | (upto - 1u)) : kFullMask;       // lanes 0 .. first total
      const unsigned miss = none & need;
      const unsigned take = miss ? ((miss & (0u - miss)) - 1u) : need;      // lanes before the first gap
      pre += warp_sum_u64((take >> lane) & 1u ? (s & kTileValue) : 0ull);
      if (total && !miss) break;
      end -= __popc(take);
      if (take == 0u) {
        const bool over = __any_sync(kFullMask, lane == 0 && wait_over(++polls, flags));
        if (over) {
          ok = false;
          break;
        }
      }
    }
    if (lane == 0) {
      if (ok && tile > 0) st_relaxed(&state[tile], kTileTotal | (pre + sum));
      pre_sh = pre;
      ok_sh = ok ? 1 : 0;
    }
  }
  __syncthreads();
  *prefix = pre_sh;
  return ok_sh != 0;
}

// ------------------------------------------------------------------ radix sort
// Keys are 64-bit, values 32-bit, digits 8 bits. The caller's key kernel
// writes the keys and counts every digit of the sort at once (DigitCounts);
// each digit is then one pass over the keys and one launch, where a histogram
// kernel, a three-kernel scan of the per-tile histograms and a scatter kernel
// took two reads and five launches. Whole builds on GB300, with the first
// pass, the digit counts and the row entries fused as in prep.cu: 20k edges
// 424 -> 188 us, 2M with repeated pairs 1.55 -> 0.84 ms, 20M 3.72 -> 3.02 ms,
// 300M 47.5 -> 41.4 ms. Tiles of 512 threads x 8 keys, two CTAs per SM, were
// the best of 256 x 8, 256 x 12, 256 x 16, 384 x 8 and 512 x 8 with one CTA
// (20M: 3.21, 3.10, 3.06, 3.18 and 3.50 ms).
#ifndef DBBC_RS_THREADS
#define DBBC_RS_THREADS 512
#endif
#ifndef DBBC_RS_ITEMS
#define DBBC_RS_ITEMS 8
#endif
#ifndef DBBC_RS_CTAS
#define DBBC_RS_CTAS 2
#endif
constexpr int kRsThreads = DBBC_RS_THREADS;
constexpr int kRsWarps = kRsThreads / 32;
constexpr int kRsItems = DBBC_RS_ITEMS;         // keys per thread
constexpr int kRsTile = kRsThreads * kRsItems;  // keys per tile
constexpr int kRsMaxPasses = 8;
static_assert(kRsThreads >= 256, "one thread per digit");

__device__ __forceinline__ uint32_t rs_digit(uint64_t key, int shift) { return (uint32_t)(key >> shift) & 0xFFu; }

inline int radix_passes(int begin_bit, int end_bit) {
  return std::max(1, ceil_div(end_bit - begin_bit, 8));
}
inline int64_t radix_tiles(int64_t n) { return ceil_div<int64_t>(std::max<int64_t>(n, 1), kRsTile); }

// Zeroed device words of one sort: digit counts of every pass, tile counters
// and tile states (see radix_pass_kernel).
struct RadixState {
  uint32_t* hist;      // [passes][256]
  unsigned* counters;  // [passes]
  uint32_t* state;     // [passes][tiles][256]
};

// Counts of all digits of a sort, kept in shared memory by the kernel that
// makes the keys. Every thread of the CTA calls start and finish.
struct DigitCounts {
  uint32_t (*h)[256];
  int passes, begin_bit;
  __device__ __forceinline__ void start() {
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x) (&h[0][0])[i] = 0;
    __syncthreads();
  }
  __device__ __forceinline__ void add(uint64_t key) {
    for (int p = 0; p < passes; p++) atomicAdd(&h[p][rs_digit(key, begin_bit + 8 * p)], 1u);
  }
  __device__ __forceinline__ void finish(uint32_t* hist) {
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x) {
      const uint32_t c = (&h[0][0])[i];
      if (c) atomicAdd(&hist[i], c);
    }
  }
};

// Where a pass's keys (and values) come from: the arrays of the pass before,
// or a transformation of another list (see prep.cu).
struct PlainLoad {
  const uint64_t* kin;
  const uint32_t* vin;
  __device__ __forceinline__ uint64_t key(uint32_t i) const { return kin[i]; }
  __device__ __forceinline__ uint32_t val(uint32_t i) const { return vin[i]; }
};

// What a pass writes: keys and / or values, and with AUX (key & aux_mask) as a
// 32-bit word per key.
struct PassOut {
  uint64_t* key;
  uint32_t* val;
  uint32_t* aux;
  uint64_t aux_mask;
};

// The lanes of the warp whose digit d equals this lane's, among the lanes of
// `valid`: one ballot per bit of d, each lane keeping the lanes that agree with
// it on that bit (a warp match instruction per key runs slower).
__device__ __forceinline__ unsigned rs_peers(uint32_t d, unsigned valid) {
  unsigned peers = valid;
#pragma unroll
  for (int b = 0; b < 8; b++) {
    const bool bit = (d >> b) & 1u;
    const unsigned bal = __ballot_sync(kFullMask, bit);
    peers &= bit ? bal : ~bal;
  }
  return peers;
}

// One digit pass of the stable sort, one tile per CTA. The tile's keys are
// loaded, kRsItems per thread in flight together; each warp ranks its keys in
// input order (digit peers per key, per-warp digit counters); the tile's digit
// counts are published, the tile is staged in shared memory in digit order,
// and thread d looks back over the earlier tiles for digit d, four of them per
// round of loads. The tile is then written out as whole digit runs. A tile
// state is one word per digit: 0 (nothing yet), 1 + the tile's count, or
// kDigitTotal | the running total (totals are below 2^31). A pass over 20M keys
// takes 157 us (1.76 TB/s; the two kernels it replaces, 70 + 100 us and their
// scan 25): 52% of the issue slots, half of them the digit ballots, the rest
// waits at the tile's barriers with 32 warps per SM.
constexpr uint32_t kDigitTotal = 0x80000000u;

template <class Load, bool HAS_V, bool WRITE_K, bool AUX>
__global__ void __launch_bounds__(kRsThreads, DBBC_RS_CTAS)
    radix_pass_kernel(Load load, PassOut out, int64_t n, int shift, const uint32_t* __restrict__ hist, uint32_t* state,
                      unsigned* counter, unsigned* flags) {
  extern __shared__ __align__(16) unsigned char rs_smem[];
  // warp digit counters first, then the staged tile, in the same memory
  uint32_t* wh = reinterpret_cast<uint32_t*>(rs_smem);
  uint64_t* sk = reinterpret_cast<uint64_t*>(rs_smem);
  uint32_t* sv = reinterpret_cast<uint32_t*>(sk + kRsTile);
  __shared__ uint32_t bstart[256], gofs[256];
  __shared__ uint32_t tot_sh;
  __shared__ int ok_sh;
  for (int i = threadIdx.x; i < kRsWarps * 256; i += kRsThreads) wh[i] = 0;
  if (threadIdx.x == 0) ok_sh = 1;
  const int64_t tile = take_tile(counter, flags);
  if (tile < 0) return;
  const int w = threadIdx.x >> 5;
  const unsigned lane = lane_id();
  const uint32_t nk = (uint32_t)n;  // below 2^31, so tiles end below 2^32
  const uint32_t tile_base = (uint32_t)tile * kRsTile;
  const uint32_t wbase = tile_base + (uint32_t)w * (kRsItems * 32) + lane;
  uint64_t key[kRsItems];
  uint32_t val[kRsItems];
#pragma unroll
  for (int j = 0; j < kRsItems; j++) {
    const uint32_t i = wbase + j * 32;
    const bool valid = i < nk;
    key[j] = valid ? load.key(i) : 0ull;
    if (HAS_V) val[j] = valid ? load.val(i) : 0u;
  }
  // exclusive prefix of the digit's count over smaller digits
  const uint32_t digit_base =
      block_excl_scan<uint32_t, kRsThreads>(threadIdx.x < 256 ? hist[threadIdx.x] : 0u, &tot_sh);

  // rank within the warp, item by item in input order
  const unsigned lt_mask = (1u << lane) - 1u;
  uint32_t loc[kRsItems];
#pragma unroll
  for (int j = 0; j < kRsItems; j++) {
    const bool ok = wbase + j * 32 < nk;
    const unsigned valid = __ballot_sync(kFullMask, ok);
    const uint32_t d = rs_digit(key[j], shift);
    const unsigned peers = rs_peers(d, valid);
    uint32_t pre = 0;
    if (ok) pre = wh[w * 256 + d];
    __syncwarp();
    loc[j] = pre + __popc(peers & lt_mask);
    if (ok && (int)lane == 31 - __clz(peers)) wh[w * 256 + d] = pre + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  {  // per digit: exclusive prefix over warps, then over digits
    const int d = threadIdx.x;
    uint32_t run = 0;
    if (d < 256) {
#pragma unroll
      for (int ww = 0; ww < kRsWarps; ww++) {
        const uint32_t c = wh[ww * 256 + d];
        wh[ww * 256 + d] = run;
        run += c;
      }
      st_relaxed(&state[tile * 256 + d], tile == 0 ? kDigitTotal | run : 1u + run);
    }
    const uint32_t ex = block_excl_scan<uint32_t, kRsThreads>(run, &tot_sh);
    if (d < 256) {
      bstart[d] = ex;
      gofs[d] = run;  // the tile's count, until the look-back
    }
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kRsItems; j++) {
    const uint32_t d = rs_digit(key[j], shift);
    loc[j] += bstart[d] + wh[w * 256 + d];
  }
  __syncthreads();  // the counters' memory is free
#pragma unroll
  for (int j = 0; j < kRsItems; j++) {
    if (wbase + j * 32 < nk && DBBC_CHECK(loc[j] < (uint32_t)kRsTile)) {
      sk[loc[j]] = key[j];
      if (HAS_V) sv[loc[j]] = val[j];
    }
  }
  if (threadIdx.x < 256) {  // look back for digit d
    const int d = threadIdx.x;
    const uint32_t count = gofs[d];
    uint32_t before = 0, polls = 0;
    bool ok = may_wait(tile, flags);
    for (int64_t t = tile - 1; ok && t >= 0;) {
      uint32_t s[4];
#pragma unroll
      for (int k = 0; k < 4; k++) s[k] = t - k >= 0 ? ld_relaxed(&state[(t - k) * 256 + d]) : kDigitTotal;
      int used = 0;
      bool done = false;
#pragma unroll
      for (int k = 0; k < 4; k++) {
        if (!done && used == k && s[k] != 0u) {
          used = k + 1;
          done = (s[k] & kDigitTotal) != 0u;
          before += done ? s[k] & ~kDigitTotal : s[k] - 1u;
        }
      }
      if (done) break;
      t -= used;
      if (used == 0 && wait_over(++polls, flags)) {
        ok = false;
        break;
      }
    }
    if (ok) {
      if (tile > 0) st_relaxed(&state[tile * 256 + d], kDigitTotal | (before + count));
    } else {
      ok_sh = 0;
    }
    gofs[d] = digit_base + before - bstart[d];
  }
  __syncthreads();
  if (!ok_sh) return;
  const uint32_t cnt = min(nk - tile_base, (uint32_t)kRsTile);
#pragma unroll
  for (int j = 0; j < kRsItems; j++) {
    const uint32_t i = threadIdx.x + j * kRsThreads;
    if (i < cnt) {
      const uint64_t k = sk[i];
      const uint32_t g = gofs[rs_digit(k, shift)] + i;
      if (g < nk) {
        if (WRITE_K) out.key[g] = k;
        if (HAS_V) out.val[g] = sv[i];
        if (AUX) out.aux[g] = (uint32_t)(k & out.aux_mask);
      } else {
        (void)DBBC_CHECK(false);  // checked builds: recorded
      }
    }
  }
}

// Sort digit of an estimate x >= 1, larger ones first, in 2^log_steps steps per
// octave: the top bits of x as a float. Work lists are ordered by it for LPT
// scheduling, which needs no finer order (one digit pass sorts them).
__device__ __forceinline__ uint32_t estimate_digit(uint32_t x, int log_steps, uint32_t digits) {
  const uint32_t q = (__float_as_uint((float)x) >> (23 - log_steps)) - (127u << log_steps);
  return digits - 1u - min(q, digits - 1u);
}

// Launch one pass (pass number `pass` of the sort: digit counts, tile counter
// and states of `st`).
template <class Load, bool HAS_V, bool WRITE_K, bool AUX>
void radix_pass(const Load& load, const PassOut& out, int64_t n, int begin_bit, int pass, const RadixState& st,
                unsigned* flags, cudaStream_t s) {
  auto fn = radix_pass_kernel<Load, HAS_V, WRITE_K, AUX>;
  const size_t staged = (size_t)kRsTile * (8 + (HAS_V ? 4 : 0)), counters = (size_t)kRsWarps * 256 * 4;
  const size_t smem = std::max(staged, counters);
  (void)resident_ctas((const void*)fn, kRsThreads, smem, smem);
  const int64_t tiles = radix_tiles(n);
  launch_overlapped(fn, tiles, kRsThreads, smem, s, load, out, n, begin_bit + 8 * pass, st.hist + 256 * pass,
                    st.state + (size_t)pass * tiles * 256, st.counters + pass, flags);
}

// dst[i] = src[idx[i]]: a list in the order that a sort found.
template <typename T>
__global__ void gather_kernel(const T* __restrict__ src, const uint32_t* __restrict__ idx, int64_t n,
                              T* __restrict__ dst, const unsigned* flags) {
  if (cta_stopped(flags)) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t j = idx[i];
    if (DBBC_CHECK((int64_t)j < n)) dst[i] = src[j];
  }
}

}  // namespace dbbc
