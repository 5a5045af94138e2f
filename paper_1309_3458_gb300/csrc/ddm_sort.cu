// LSD radix sort of 64-bit words: keys packed above their ids, or keys with a
// 32-bit payload.
//
// Sorts the subscriptions into the interval tree order of Section IV (by lower
// bound, ties then put in the order of the upper bound, remaining ties in id
// order), and the updates and the re-sorts into locality orders.  Three
// forms by size, each a stable sort over 8-bit digits:
//   * up to 16 tiles of 2,048 keys: one thread-block cluster keeps the keys
//     in distributed shared memory for every pass (k_sort_cluster);
//   * up to one resident tile per SM: one cooperative launch runs every pass,
//     the tiles exchanging digit counts across bounded grid barriers
//     (k_sort_grid);
//   * beyond: onesweep, after Adinets & Merrill
//     ("Onesweep", 2022): one histogram pass over the keys computes all
//     digit histograms at once, a tiny kernel scans them into digit
//     bases, and each digit pass is ONE kernel: a CTA takes the next tile
//     (ticket from an atomic counter, so every earlier tile is already
//     resident), ranks its keys per digit with a warp match (one ballot per
//     digit bit) and per-warp counters, publishes its per-digit counts,
//     resolves its global per-digit offsets by decoupled look-back over
//     earlier tiles, and scatters through shared memory so that global
//     stores come out as runs of equal digits.
// Every wait is bounded: after kSpinLimit polls a CTA records kErrTimeout and
// carries on (look-back) or returns (grid barrier), so the kernels always
// terminate.
#include <algorithm>
#include <atomic>

#include "ddm_internal.cuh"

namespace ddm {
namespace {

constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kPasses = 64 / kRadixBits;
constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = kSortTile / kThreads;  // 16 keys per thread
constexpr uint32_t kFlagAgg = 1u << 30;       // tile aggregate available
constexpr uint32_t kFlagInc = 2u << 30;       // inclusive prefix available
constexpr uint32_t kFlagMask = 3u << 30;
constexpr uint32_t kValMask = (1u << 30) - 1;
constexpr uint32_t kSpinLimit = 1u << 22;

static_assert(kSortTile % kThreads == 0, "tile must split evenly over threads");

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t r;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
  return r;
}

// Lanes of the warp holding the same digit: one ballot per digit bit.
// Measured: an 8,192-key single-CTA sort took 59 instead of 88 us with this in
// place of match.any, which the SM's warps issue one at a time.
__device__ __forceinline__ uint32_t same_digit_lanes(uint32_t dig) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < kRadixBits; ++b) {
    const uint32_t bit = (dig >> b) & 1u;
    const uint32_t votes = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? votes : ~votes;
  }
  return peers;
}

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Bounded poll of a look-back word: returns it once any bit of `mask` is
// set, or 0 with *timed_out after `limit` polls (64 ns apart), so that no
// wait can outlive a predecessor that never publishes.
__device__ __forceinline__ uint32_t poll_flag(const uint32_t* p, uint32_t mask, uint32_t limit,
                                              bool* timed_out) {
  for (uint32_t spins = 0;; ++spins) {
    const uint32_t w = ld_relaxed(p);
    if (w & mask) return w;
    if (spins >= limit) {
      *timed_out = true;
      return 0u;
    }
    __nanosleep(64);
  }
}

// A packed word: the key above the id (id_bits wide), so that a pass moves
// one 8-byte word per element where keys and ids in separate arrays are
// twelve bytes in two streams.  The first pass builds the words of a source
// (SortSource): k32[i], with hi[i] above it, and the position as id.
__device__ __forceinline__ unsigned long long source_word(const SortSource& src, uint32_t i) {
  unsigned long long k = __ldg(src.k32 + i);
  if (src.hi) k |= (unsigned long long)__ldg(src.hi + i) << src.k32_bits;
  return (k << src.id_bits) | i;
}

// The first words of a sort by both keys, and those rebuilt between the two.
__device__ __forceinline__ unsigned long long second_word(const SortSource& src, uint32_t i) {
  return ((unsigned long long)float_key(__ldg(src.second + i)) << src.id_bits) | i;
}
__device__ __forceinline__ unsigned long long first_word(const SortSource& src, unsigned long long w) {
  const uint32_t id = (uint32_t)(w & ((1ull << src.id_bits) - 1ull));
  return ((unsigned long long)__ldg(src.k32 + id) << src.id_bits) | id;
}

// Test hook for the bounded waits: poll a word nothing sets.
__global__ void k_debug_wait(const uint32_t* __restrict__ word, uint32_t limit,
                             Status* __restrict__ st) {
  bool timed_out = false;
  poll_flag(word, kFlagMask, limit, &timed_out);
  if (timed_out && threadIdx.x == 0) atomicOr(&st->err, kErrTimeout);
}

// All eight digit histograms in one read of the keys.
__global__ void __launch_bounds__(kThreads)
k_histogram(const unsigned long long* __restrict__ keys, uint32_t n, uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kPasses * kRadix];
  for (int t = threadIdx.x; t < kPasses * kRadix; t += kThreads) h[t] = 0;
  __syncthreads();
  const uint32_t stride = gridDim.x * kThreads;
  for (uint32_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += stride) {
    const unsigned long long k = keys[i];
#pragma unroll
    for (int p = 0; p < kPasses; ++p)
      atomicAdd(&h[p * kRadix + (uint32_t)((k >> (p * kRadixBits)) & (kRadix - 1))], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kPasses * kRadix; t += kThreads)
    if (h[t]) atomicAdd(&hist[t], h[t]);
}

// Exclusive scan of each pass's 256-bin histogram, in place (one CTA per pass).
__global__ void __launch_bounds__(kRadix) k_hist_scan(uint32_t* __restrict__ hist) {
  __shared__ uint32_t warp_tot[kRadix / 32];
  uint32_t* h = hist + blockIdx.x * kRadix;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const uint32_t v = h[t];
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  uint32_t pre = 0;
  for (int i = 0; i < w; ++i) pre += warp_tot[i];
  h[t] = pre + x - v;
}

struct OnesweepSmem {
  uint32_t whist[kWarps][kRadix];  // per-warp digit counts, then per-warp exclusive offsets
  uint32_t lstart[kRadix];         // tile-local start of each digit
  uint32_t gbase[kRadix];          // global position of local slot 0 of each digit
  uint32_t wtot[kRadix / 32];
  uint32_t tile;
  unsigned long long keys[kSortTile];
  uint32_t vals[kSortTile];
};

// Three resident CTAs per SM (registers capped at 80, a few spilled): measured
// faster than two CTAs at 128 registers.
__global__ void __launch_bounds__(kThreads, 3)
k_onesweep(const unsigned long long* __restrict__ in_keys, const uint32_t* __restrict__ in_vals,
           unsigned long long* __restrict__ out_keys, uint32_t* __restrict__ out_vals, uint32_t n,
           int shift, const uint32_t* __restrict__ digit_base, uint32_t* __restrict__ lookback,
           uint32_t* __restrict__ counter, Status* __restrict__ st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  OnesweepSmem& sm = *reinterpret_cast<OnesweepSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  if (tid == 0) sm.tile = atomicAdd(counter, 1u);
  for (int t = tid; t < kWarps * kRadix; t += kThreads) (&sm.whist[0][0])[t] = 0;
  __syncthreads();
  const uint32_t tile = sm.tile;
  const size_t tile_base = (size_t)tile * kSortTile;
  const uint32_t tile_valid = (uint32_t)min((size_t)kSortTile, (size_t)n - tile_base);

  // Load: warp w owns keys [w*512, w*512+512) of the tile; item i of a lane
  // is key w*512 + i*32 + lane, so (warp, item, lane) is input order.
  unsigned long long key[kItems];
  uint32_t val[kItems], dig[kItems], rank[kItems];
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t local = warp * (kItems * 32) + i * 32 + lane;
    if (local < tile_valid) {
      key[i] = in_keys[tile_base + local];
      val[i] = in_vals[tile_base + local];
      dig[i] = (uint32_t)(key[i] >> shift) & (kRadix - 1);
    } else {  // padding: the largest key, so it ranks last and its slots go unused
      key[i] = ~0ull;
      val[i] = 0;
      dig[i] = kRadix - 1;
    }
  }

  // Rank within the warp, item by item: lanes sharing a digit are found by
  // ballots; the lowest such lane bumps the warp's counter for the digit.
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t peers = same_digit_lanes(dig[i]);
    const uint32_t before = sm.whist[warp][dig[i]];
    rank[i] = before + __popc(peers & lt);
    __syncwarp();
    if ((peers & lt) == 0) sm.whist[warp][dig[i]] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();

  // Thread t owns digit t: per-warp exclusive offsets and the tile count.
  uint32_t count = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    const uint32_t c = sm.whist[w][tid];
    sm.whist[w][tid] = count;
    count += c;
  }
  uint32_t* my_slot = lookback + (size_t)tile * kRadix + tid;
  st_relaxed(my_slot, (tile == 0 ? kFlagInc : kFlagAgg) | count);

  // Tile-local exclusive scan of the digit counts.
  uint32_t x = count;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sm.wtot[warp] = x;
  __syncthreads();
  uint32_t pre = 0;
  for (int w = 0; w < warp; ++w) pre += sm.wtot[w];
  const uint32_t lstart = pre + x - count;
  sm.lstart[tid] = lstart;

  // Decoupled look-back over earlier tiles for digit `tid`.
  uint32_t excl = 0;
  if (tile > 0) {
    uint32_t p = tile - 1;
    for (;;) {
      bool timed_out = false;
      const uint32_t w = poll_flag(lookback + (size_t)p * kRadix + tid, kFlagMask, kSpinLimit,
                                   &timed_out);
      if (timed_out) {
        atomicOr(&st->err, kErrTimeout);
        break;
      }
      excl += w & kValMask;
      if ((w & kFlagMask) == kFlagInc || p == 0) break;
      --p;
    }
    st_relaxed(my_slot, kFlagInc | (excl + count));
  }
  sm.gbase[tid] = digit_base[tid] + excl - lstart;  // modular: gbase + slot is exact
  __syncthreads();

  // Scatter into shared memory in (digit, input order) order ...
#pragma unroll
  for (int i = 0; i < kItems; ++i) {
    const uint32_t slot = sm.lstart[dig[i]] + sm.whist[warp][dig[i]] + rank[i];
    sm.keys[slot] = key[i];
    sm.vals[slot] = val[i];
  }
  __syncthreads();
  // ... and out to global memory, consecutive threads taking consecutive slots.
  for (uint32_t s = tid; s < tile_valid; s += kThreads) {
    const unsigned long long k = sm.keys[s];
    const uint32_t g = sm.gbase[(uint32_t)(k >> shift) & (kRadix - 1)] + s;
    if (DDM_IN_BOUNDS(g < n, st)) {
      out_keys[g] = k;
      out_vals[g] = sm.vals[s];
    }
  }
}

// Digit histograms of a packed sort, in one read of its source (or words).
// Bound by the shared-memory atomics (107 us for 2.5e7 keys of three digits).
// The digits of a warp's elements are often all equal (high digits, instance
// numbers): then one lane adds them at once, where 32 atomics on one word
// would take 32 turns.
// TWO: the second key's digits too (behind the first's) if the sort is by both.
template <bool TWO>
__global__ void __launch_bounds__(kThreads)
k_histogram_packed(const unsigned long long* __restrict__ words, SortSource src, uint32_t n,
                   int passes, uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[kPasses * kRadix];
  const bool both = TWO && *src.both;
  const int total = both ? 2 * passes : passes;
  for (int t = threadIdx.x; t < total * kRadix; t += kThreads) h[t] = 0;
  __syncthreads();
  const uint32_t stride = gridDim.x * kThreads;
  const int lane = threadIdx.x & 31;
  for (size_t i0 = blockIdx.x * kThreads + (threadIdx.x & ~31u); i0 < n; i0 += (size_t)stride * 4) {
    unsigned long long k[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t i = i0 + (size_t)u * stride + lane;
      k[u] = i >= n ? 0ull : (src.k32 ? source_word(src, (uint32_t)i) : words[i]) >> src.id_bits;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const size_t first = i0 + (size_t)u * stride;
      const bool whole = first + 32u <= n;  // warp-uniform
      if (!whole && first + lane >= n) continue;
      for (int p = 0; p < passes; ++p) {
        const uint32_t d = (uint32_t)(k[u] >> (p * kRadixBits)) & (kRadix - 1);
        if (whole && __all_sync(0xffffffffu, d == __shfl_sync(0xffffffffu, d, 0))) {
          if (lane == 0) atomicAdd(&h[p * kRadix + d], 32u);
        } else {
          atomicAdd(&h[p * kRadix + d], 1u);
        }
      }
    }
  }
  if (TWO && both) {
    for (size_t i = blockIdx.x * kThreads + threadIdx.x; i < n; i += stride) {
      const uint32_t k = float_key(__ldg(src.second + i));
      for (int p = 0; p < passes; ++p)
        atomicAdd(&h[(passes + p) * kRadix + ((k >> (p * kRadixBits)) & (kRadix - 1))], 1u);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < total * kRadix; t += kThreads)
    if (h[t]) atomicAdd(&hist[t], h[t]);
}

// The onesweep pass on packed words: 512 threads with eight words each, so
// that three CTAs fit an SM in 40 registers (the pass on keys and ids needs 80
// and spills), half the words per thread to wait for and to rank in turn, one
// scattered stream instead of two.  FROM: where the words come from (kFromFirst:
// the source, or, between the two halves of a sort by both keys, rebuilt; the
// passes of kFromSecond's half, `second_half`, do nothing otherwise); LAST:
// only the ids go out (as from the `final` pass of a sort by both keys).
constexpr int kPackThreads = 512;
constexpr int kPackWarps = kPackThreads / 32;
constexpr int kPackItems = kSortTile / kPackThreads;  // 8

struct PackedSmem {
  uint32_t whist[kPackWarps][kRadix];
  uint32_t lstart[kRadix];
  uint32_t gbase[kRadix];
  uint32_t wtot[kRadix / 32];
  uint32_t tile;
  unsigned long long words[kSortTile];
};

enum { kFromWords, kFromFirst, kFromSecond };
template <int FROM, bool LAST>
__global__ void __launch_bounds__(kPackThreads, 3)
k_onesweep_packed(const unsigned long long* __restrict__ in, SortSource src,
                  unsigned long long* __restrict__ out, uint32_t* __restrict__ out_ids, uint32_t n,
                  int shift, const uint32_t* __restrict__ digit_base,
                  uint32_t* __restrict__ lookback, uint32_t* __restrict__ counter,
                  bool second_half, bool final, Status* __restrict__ st) {
  const bool both = (second_half || final || FROM == kFromFirst) && src.both && *src.both;
  if (second_half && !both) return;
  const bool ids = final && both;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PackedSmem& sm = *reinterpret_cast<PackedSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt();
  if (tid == 0) sm.tile = atomicAdd(counter, 1u);
  for (int t = lane; t < kRadix; t += 32) sm.whist[warp][t] = 0;
  __syncthreads();
  const uint32_t tile = sm.tile;
  const uint32_t base = tile * (uint32_t)kSortTile;
  const uint32_t valid = min((uint32_t)kSortTile, n - base);
  unsigned long long word[kPackItems];
  uint32_t rank[kPackItems];
#pragma unroll
  for (int i = 0; i < kPackItems; ++i) {
    const uint32_t local = warp * (kPackItems * 32) + i * 32 + lane;
    if (local >= valid)
      word[i] = ~0ull;
    else if (FROM == kFromSecond)
      word[i] = second_word(src, base + local);
    else if (FROM == kFromFirst)
      word[i] = both ? first_word(src, in[base + local]) : source_word(src, base + local);
    else
      word[i] = in[base + local];
  }
#pragma unroll
  for (int i = 0; i < kPackItems; ++i) {
    const uint32_t d = (uint32_t)(word[i] >> shift) & (kRadix - 1);
    const uint32_t peers = same_digit_lanes(d);
    const uint32_t before = sm.whist[warp][d];
    rank[i] = before + __popc(peers & lt);
    __syncwarp();
    if ((peers & lt) == 0) sm.whist[warp][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // Thread t < 256 owns digit t: per-warp first slots, the tile's count, its
  // first slot in the tile and (look-back) in the output.
  uint32_t count = 0, x = 0;
  uint32_t* my_slot = lookback + (size_t)tile * kRadix + tid;
  if (tid < kRadix) {
#pragma unroll
    for (int w = 0; w < kPackWarps; ++w) {
      const uint32_t c = sm.whist[w][tid];
      sm.whist[w][tid] = count;
      count += c;
    }
    st_relaxed(my_slot, (tile == 0 ? kFlagInc : kFlagAgg) | count);
    x = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) sm.wtot[warp] = x;
  }
  __syncthreads();
  if (tid < kRadix) {
    uint32_t pre = 0;
    for (int w = 0; w < warp; ++w) pre += sm.wtot[w];
    const uint32_t lstart = pre + x - count;
    sm.lstart[tid] = lstart;
    uint32_t excl = 0;
    if (tile > 0) {
      uint32_t p = tile - 1;
      for (;;) {
        bool timed_out = false;
        const uint32_t w = poll_flag(lookback + (size_t)p * kRadix + tid, kFlagMask, kSpinLimit,
                                     &timed_out);
        if (timed_out) {
          atomicOr(&st->err, kErrTimeout);
          break;
        }
        excl += w & kValMask;
        if ((w & kFlagMask) == kFlagInc || p == 0) break;
        --p;
      }
      st_relaxed(my_slot, kFlagInc | (excl + count));
    }
    sm.gbase[tid] = digit_base[tid] + excl - lstart;  // modular: gbase + slot is exact
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kPackItems; ++i) {
    const uint32_t d = (uint32_t)(word[i] >> shift) & (kRadix - 1);
    sm.words[sm.lstart[d] + sm.whist[warp][d] + rank[i]] = word[i];
  }
  __syncthreads();
  for (uint32_t q = tid; q < valid; q += kPackThreads) {
    const unsigned long long k = sm.words[q];
    const uint32_t g = sm.gbase[(uint32_t)(k >> shift) & (kRadix - 1)] + q;
    if (!DDM_IN_BOUNDS(g < n, st)) continue;
    if (LAST || ids)
      out_ids[g] = (uint32_t)(k & ((1ull << src.id_bits) - 1ull));
    else
      out[g] = k;
  }
}

// Ranking of one tile of 512 * ITEMS keys held in registers by 512 threads
// (positions past the set's end hold ~0: they rank last, and the slots from
// the valid count on are not written out; they are counted for digit 255,
// which has no digit and, in the last tile, no tile behind it)
// (item i of lane l in warp w is the tile's element w*32*ITEMS + i*32 + l):
// the same stable ranking as k_onesweep (warp match + per-warp counters,
// warps in order).  Afterwards whist[w][dg] is warp w's first slot within
// digit dg, lstart[dg] the digit's first slot in the tile, and the returned
// count (threads < 256, digit = thread) the tile's keys with that digit.
constexpr int kSmallThreads = 512;
constexpr int kSmallWarps = kSmallThreads / 32;

struct RankSmem {
  uint32_t whist[kSmallWarps][kRadix];
  uint32_t wtot[kRadix / 32];
  uint32_t lstart[kRadix];
};

template <int ITEMS>
__device__ __forceinline__ uint32_t rank_tile(RankSmem& sm, const unsigned long long (&key)[ITEMS],
                                              uint32_t (&rank)[ITEMS], int shift) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt();
  for (int t = lane; t < kRadix; t += 32) sm.whist[warp][t] = 0;
  __syncwarp();
  // four items' ballots first, then the serial chain through the counters
#pragma unroll
  for (int i0 = 0; i0 < ITEMS; i0 += 4) {
    uint32_t peers[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      peers[u] = same_digit_lanes((uint32_t)(key[i0 + u] >> shift) & (kRadix - 1));
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t* h = &sm.whist[warp][(uint32_t)(key[i0 + u] >> shift) & (kRadix - 1)];
      const uint32_t before = *h;
      rank[i0 + u] = before + __popc(peers[u] & lt);
      __syncwarp();
      if ((peers[u] & lt) == 0) *h = before + __popc(peers[u]);
      __syncwarp();
    }
  }
  __syncthreads();
  uint32_t count = 0;
  if (tid < kRadix) {  // thread t owns digit t: per-warp offsets, tile offsets
#pragma unroll
    for (int w = 0; w < kSmallWarps; ++w) {
      const uint32_t c = sm.whist[w][tid];
      sm.whist[w][tid] = count;
      count += c;
    }
    uint32_t x = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) sm.wtot[warp] = x;
    sm.lstart[tid] = x - count;  // within-warp part; warp prefix added below
  }
  __syncthreads();
  if (tid < kRadix) {
    uint32_t pre = 0;
    for (int w = 0; w < warp; ++w) pre += sm.wtot[w];
    sm.lstart[tid] += pre;
  }
  __syncthreads();
  return count;
}

// Mid-size arrays (up to kGridMaxTiles tiles of 512 * ITEMS keys, all CTAs
// resident): one cooperative launch runs every pass.  CTA g holds tile g in
// registers and ranks it (rank_tile); the tiles then exchange their
// digit counts through global memory across a grid barrier, each CTA takes
// its digit offsets from the counts (no look-back chain), scatters, and a
// second barrier ends the pass.  Tiles come in groups of kGridGroup: a tile
// adds its counts into its group's sums (global atomics) and stores them,
// 16-bit and packed two to a word, in its own row; a digit's total is the
// sum of the group sums and the part before tile g the sums of the groups
// before g's plus the rows of g's group before it -- at most 12 + 15 reads
// per digit instead of one per tile.  The group sums are double-buffered by
// pass parity, and each pass clears the buffer of the next.  Smaller tiles
// (fewer items per thread) spread a set over more SMs: each pass's ranking
// and scatter shrink with the tile, the two barriers do not.
constexpr uint32_t kGridMaxTiles = 192;
constexpr uint32_t kGridGroup = 16;
constexpr uint32_t kGridGroups = kGridMaxTiles / kGridGroup;  // 12
// Scratch words of a cooperative sort: the per-tile rows, the group sums of
// both parities and the barrier counter (the last two zeroed before each
// launch).
constexpr size_t kGridRowWords = (size_t)kGridMaxTiles * (kRadix / 2);
constexpr size_t kGridSumWords = 2 * (size_t)kGridGroups * kRadix;
constexpr size_t kGridScratchWords = kGridRowWords + kGridSumWords + 32;

template <int ITEMS, bool PACKED>
struct GridSortSmem {
  RankSmem r;
  uint32_t gbase[kRadix];
  uint32_t dtot[kRadix / 32];
  int abort;
  int pad[3];
  unsigned long long keys[kSmallThreads * ITEMS];
  uint32_t vals[PACKED ? 1 : kSmallThreads * ITEMS];
};

// Grid-wide barrier for a cooperative launch (all CTAs resident).  `bar` is
// zeroed before the launch and only grows; barrier number b completes when
// it reaches gridDim.x * b.  The wait is bounded: after kSpinLimit polls
// the CTA records kErrTimeout and the kernel returns false to every thread
// of it, so every CTA ends (those left waiting time out in turn).
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t target, Status* st,
                                             int* s_abort) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    bool timed_out = false;
    for (uint32_t spins = 0;; ++spins) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if (spins >= kSpinLimit) {
        timed_out = true;
        break;
      }
      __nanosleep(32);
    }
    if (timed_out) {
      atomicOr(&st->err, kErrTimeout);
      *s_abort = 1;
    }
    __threadfence();
  }
  __syncthreads();
  return *s_abort == 0;
}

// Two CTAs per SM up to 4,096-key tiles (64 registers, no spill): a one-shot
// call sorts both of its sets at the same time.
// PACKED: words (from `src` if it has a source, else keys0), the ids to vals0
// at the end; else keys and ids.
template <int ITEMS, bool PACKED>
__global__ void __launch_bounds__(kSmallThreads, ITEMS <= 8 ? 2 : 1)
k_sort_grid(unsigned long long* __restrict__ keys0, uint32_t* __restrict__ vals0,
            unsigned long long* __restrict__ keys1, uint32_t* __restrict__ vals1, uint32_t n,
            int passes, SortSource src, uint32_t* __restrict__ table, uint32_t* __restrict__ bar,
            Status* __restrict__ st) {
  const bool both = PACKED && src.both && *src.both;  // every CTA alike
  const int half = passes;  // a sort by both keys: twice, the second key first
  if (both) passes = 2 * half;
  constexpr uint32_t kTile = kSmallThreads * ITEMS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GridSortSmem<ITEMS, PACKED>& sm = *reinterpret_cast<GridSortSmem<ITEMS, PACKED>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t tile = blockIdx.x, tiles = gridDim.x;
  const size_t base = (size_t)tile * kTile;
  const uint32_t valid = (uint32_t)min((size_t)kTile, (size_t)n - base);
  if (tid == 0) sm.abort = 0;
  uint32_t barriers = 0;
  unsigned long long key[ITEMS];
  uint32_t val[PACKED ? 1 : ITEMS], rank[ITEMS];
  for (int p = 0; p < passes; ++p) {
    const unsigned long long* ik = (p & 1) ? keys1 : keys0;
    const uint32_t* iv = (p & 1) ? vals1 : vals0;
    unsigned long long* ok = (p & 1) ? keys0 : keys1;
    uint32_t* ov = (p & 1) ? vals0 : vals1;
    (void)iv;
    (void)ov;
    auto at = [&](int i) { return (uint32_t)(warp * (ITEMS * 32) + i * 32 + lane); };
    if (PACKED && p == 0 && src.k32) {
      if (both) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
          key[i] = at(i) < valid ? second_word(src, (uint32_t)base + at(i)) : ~0ull;
      } else {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
          key[i] = at(i) < valid ? source_word(src, (uint32_t)base + at(i)) : ~0ull;
      }
    } else {  // written by other CTAs of this launch: read through L2, not L1
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        key[i] = at(i) < valid ? __ldcg(ik + base + at(i)) : ~0ull;
        if constexpr (!PACKED) val[i] = at(i) < valid ? __ldcg(iv + base + at(i)) : 0u;
      }
      if (both && p == half) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i)
          if (at(i) < valid) key[i] = first_word(src, key[i]);
      }
    }
    const int shift = (PACKED && p >= half ? p - half : p) * kRadixBits + (PACKED ? src.id_bits : 0);
    const uint32_t count = rank_tile<ITEMS>(sm.r, key, rank, shift);
    uint32_t* gsum = table + kGridRowWords + (size_t)(p & 1) * kGridGroups * kRadix;
    if (tid < kRadix) {  // this tile's counts: its row (two 16-bit digits per word), its group's sums
      const uint32_t next = __shfl_down_sync(0xffffffffu, count, 1);
      if ((tid & 1) == 0) __stcg(table + (size_t)tile * (kRadix / 2) + tid / 2, count | (next << 16));
      if (count) atomicAdd(&gsum[(tile / kGridGroup) * kRadix + tid], count);
    }
    if (!grid_barrier(bar, tiles * ++barriers, st, &sm.abort)) return;
    {  // clear the next pass's group sums (last read in the previous pass)
      uint32_t* other = table + kGridRowWords + (size_t)((p + 1) & 1) * kGridGroups * kRadix;
      for (uint32_t q = tile * kSmallThreads + tid; q < kGridGroups * kRadix; q += tiles * kSmallThreads)
        other[q] = 0u;
    }
    if (tid < kRadix) {  // digit tid: its total, and the part before this tile
      const uint32_t groups = (tiles + kGridGroup - 1) / kGridGroup, mine = tile / kGridGroup;
      uint32_t tot = 0, pre = 0;
      for (uint32_t g = 0; g < groups; ++g) {
        const uint32_t c = __ldcg(gsum + g * kRadix + tid);
        tot += c;
        pre += g < mine ? c : 0u;
      }
      for (uint32_t t = mine * kGridGroup; t < tile; ++t)
        pre += (__ldcg(table + (size_t)t * (kRadix / 2) + tid / 2) >> ((tid & 1) * 16)) & 0xffffu;
      // exclusive scan of the digit totals: the digit's first position
      uint32_t x = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) sm.dtot[warp] = x;
      sm.gbase[tid] = x - tot + pre - sm.r.lstart[tid];
    }
    __syncthreads();
    if (tid < kRadix) {
      uint32_t pre = 0;
      for (int w = 0; w < warp; ++w) pre += sm.dtot[w];
      sm.gbase[tid] += pre;  // modular: gbase + slot is exact
    }
    // stage the tile in (digit, input order) order ...
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const uint32_t dg = (uint32_t)(key[i] >> shift) & (kRadix - 1);
      const uint32_t slot = sm.r.lstart[dg] + sm.r.whist[warp][dg] + rank[i];
      sm.keys[slot] = key[i];
      if constexpr (!PACKED) sm.vals[slot] = val[i];
    }
    __syncthreads();
    // ... and out, consecutive threads taking consecutive slots
    for (uint32_t q = tid; q < valid; q += kSmallThreads) {
      const unsigned long long k = sm.keys[q];
      const uint32_t g = sm.gbase[(uint32_t)(k >> shift) & (kRadix - 1)] + q;
      if (!DDM_IN_BOUNDS(g < n, st)) continue;
      if constexpr (PACKED) {
        if (p + 1 < passes || (src.words_out && !both))
          ok[g] = k;
        else
          vals0[g] = (uint32_t)(k & ((1ull << src.id_bits) - 1ull));
      } else {
        ok[g] = k;
        ov[g] = sm.vals[q];
      }
    }
    if (p + 1 < passes && !grid_barrier(bar, tiles * ++barriers, st, &sm.abort)) return;
  }
}

// Small sets (up to kClusterMax tiles of 512 * ITEMS keys): one thread-block
// cluster holds the whole set in shared memory.  Each pass ranks a tile as
// k_sort_grid does, writes its digit counts into every CTA's count table
// (distributed shared memory), and after a cluster barrier scatters its
// keys straight into the shared-memory tiles of their next owners; a second
// cluster barrier ends the pass, and only the last pass writes to global
// memory.  Both barriers are the hardware cluster barrier (no polling), and
// no key goes through L2 between passes.
constexpr uint32_t kClusterMax = 16;

template <int ITEMS, bool PACKED>
struct ClusterSortSmem {
  RankSmem r;
  uint32_t gbase[kRadix];
  uint32_t dtot[kRadix / 32];
  uint32_t table[kClusterMax][kRadix];  // row j: CTA j's digit counts
  unsigned long long tile_k[kSmallThreads * ITEMS];  // this CTA's keys of the next pass
  uint32_t tile_v[PACKED ? 1 : kSmallThreads * ITEMS];
  unsigned long long stage_k[kSmallThreads * ITEMS];  // this pass's keys in digit order
  uint32_t stage_v[PACKED ? 1 : kSmallThreads * ITEMS];
};

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;"
               ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address of `p` (this CTA's shared memory) in CTA `cta`'s shared memory.
__device__ __forceinline__ uint32_t remote_smem(const void* p, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
               : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(cta));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void st_remote(uint32_t a, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

template <int ITEMS, bool PACKED>
__global__ void __launch_bounds__(kSmallThreads, 1)
k_sort_cluster(const unsigned long long* __restrict__ in_k, const uint32_t* __restrict__ in_v,
               unsigned long long* __restrict__ out_k, uint32_t* __restrict__ out_v, uint32_t n,
               int passes, SortSource src) {
  const bool both = PACKED && src.both && *src.both;  // every CTA alike
  const int half = passes;
  if (both) passes = 2 * half;
  constexpr uint32_t kTile = kSmallThreads * ITEMS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ClusterSortSmem<ITEMS, PACKED>& sm = *reinterpret_cast<ClusterSortSmem<ITEMS, PACKED>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t me = cluster_rank(), ctas = gridDim.x;  // the grid is one cluster
  const uint32_t base = me * kTile;
  const uint32_t valid = min(kTile, n - base);
  unsigned long long key[ITEMS];
  uint32_t val[PACKED ? 1 : ITEMS], rank[ITEMS];
  auto at = [&](int i) { return (uint32_t)(warp * (ITEMS * 32) + i * 32 + lane); };
  if (PACKED && src.k32) {
    if (both) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) key[i] = at(i) < valid ? second_word(src, base + at(i)) : ~0ull;
    } else {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) key[i] = at(i) < valid ? source_word(src, base + at(i)) : ~0ull;
    }
  } else {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      key[i] = at(i) < valid ? in_k[base + at(i)] : ~0ull;
      if constexpr (!PACKED) val[i] = at(i) < valid ? in_v[base + at(i)] : 0u;
    }
  }
  for (int p = 0; p < passes; ++p) {
    const int shift = (PACKED && p >= half ? p - half : p) * kRadixBits + (PACKED ? src.id_bits : 0);
    const uint32_t count = rank_tile<ITEMS>(sm.r, key, rank, shift);
    if (tid < kRadix)
      for (uint32_t j = 0; j < ctas; ++j) st_remote(remote_smem(&sm.table[me][tid], j), count);
    cluster_sync_all();  // every table complete; every CTA holds its keys in registers
    if (tid < kRadix) {  // the digit's first position, plus the CTAs before this one
      uint32_t tot = 0, pre = 0;
      for (uint32_t j = 0; j < ctas; ++j) {
        const uint32_t c = sm.table[j][tid];
        tot += c;
        pre += j < me ? c : 0u;
      }
      uint32_t x = tot;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (lane == 31) sm.dtot[warp] = x;
      sm.gbase[tid] = x - tot + pre - sm.r.lstart[tid];
    }
    __syncthreads();
    if (tid < kRadix) {
      uint32_t pre = 0;
      for (int w = 0; w < warp; ++w) pre += sm.dtot[w];
      sm.gbase[tid] += pre;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const uint32_t dg = (uint32_t)(key[i] >> shift) & (kRadix - 1);
      const uint32_t slot = sm.r.lstart[dg] + sm.r.whist[warp][dg] + rank[i];
      sm.stage_k[slot] = key[i];
      if constexpr (!PACKED) sm.stage_v[slot] = val[i];
    }
    __syncthreads();
    const bool last = p + 1 == passes;
    // consecutive threads take consecutive slots: runs of one digit land in
    // consecutive positions of one owner
    for (uint32_t q = tid; q < valid; q += kSmallThreads) {
      const unsigned long long k = sm.stage_k[q];
      const uint32_t g = sm.gbase[(uint32_t)(k >> shift) & (kRadix - 1)] + q;
      if (!DDM_IN_BOUNDS(g < n, nullptr)) continue;
      if (last) {
        if constexpr (PACKED) {
          if (src.words_out && !both)
            out_k[g] = k;
          else
            out_v[g] = (uint32_t)(k & ((1ull << src.id_bits) - 1ull));
        } else {
          out_k[g] = k;
          out_v[g] = sm.stage_v[q];
        }
      } else {
        const uint32_t owner = g / kTile, at = g % kTile;
        st_remote(remote_smem(&sm.tile_k[at], owner), k);
        if constexpr (!PACKED) st_remote(remote_smem(&sm.tile_v[at], owner), sm.stage_v[q]);
      }
    }
    if (last) break;
    cluster_sync_all();  // every key of the next pass is in its owner's tile
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const uint32_t local = warp * (ITEMS * 32) + i * 32 + lane;
      key[i] = local < valid ? sm.tile_k[local] : ~0ull;
      if constexpr (!PACKED) val[i] = local < valid ? sm.tile_v[local] : 0u;
    }
    if (both && p + 1 == half) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i)
        if (at(i) < valid) key[i] = first_word(src, key[i]);
    }
  }
}

// The d = 1 tree's order is by lower bound, upper bound, id.  The upper bound
// matters only among equal lower bounds, so the set is sorted by the lower
// bound alone (four digits instead of eight) unless one value abounds.  Then
// every element counts those of its run (equal keys, next to it) that come
// before it, by upper bound and, ids ascending already, by position: a CTA
// stages a tile's keys and kNearRun on either side, and the upper bounds of
// those with an equal neighbour.  Bound by reading the words and writing the
// ids where few tie.  Longer runs are listed for a warp or a CTA each
// (k_long_ties).  The build of 2e7 extents in runs of 40: 2.58 ms by both
// bounds, 1.68 so; without ties 2.60 and 1.55.
constexpr uint32_t kTieTile = 1024, kTieSpan = kTieTile + 2 * kNearRun;
__global__ void __launch_bounds__(256)
k_tie_order(const unsigned long long* __restrict__ words, uint32_t n, int id_bits,
            const float* __restrict__ hi, uint32_t* __restrict__ vals, uint2* __restrict__ list,
            Status* __restrict__ st) {
  if (st->both != 0u) return;  // sorted by both bounds: the ids are there
  __shared__ uint32_t s_lo[kTieSpan], s_hi[kTieSpan];
  __shared__ uint32_t s_head[kTieSpan / 32];  // bit j: a run starts at j (or the set ends)
  const unsigned long long idm = (1ull << id_bits) - 1ull;
  constexpr int kEach = (kTieSpan + 255) / 256;
  for (uint32_t t0 = blockIdx.x * kTieTile; t0 < n; t0 += gridDim.x * kTieTile) {
    // index j of the span is position t0 + j - kNearRun; [first, last) exist
    const uint32_t first = t0 ? 0u : kNearRun, last = min(kTieSpan, n - t0 + kNearRun);
    uint32_t id[kEach];
    __syncthreads();  // the previous tile has been read
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const uint32_t j = (uint32_t)u * 256u + threadIdx.x;
      id[u] = 0u;
      if (j >= first && j < last) {
        const unsigned long long w = words[t0 + j - kNearRun];
        s_lo[j] = (uint32_t)(w >> id_bits);
        id[u] = (uint32_t)(w & idm);
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const uint32_t j = (uint32_t)u * 256u + threadIdx.x;
      if (j >= kTieSpan) break;  // whole warps
      const uint32_t heads =
          __ballot_sync(0xffffffffu, j <= first || j >= last || s_lo[j] != s_lo[j - 1u]);
      if ((threadIdx.x & 31u) == 0u) s_head[j / 32u] = heads;
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const uint32_t j = (uint32_t)u * 256u + threadIdx.x;
      if (j < first || j >= last) continue;
      const uint32_t next = j + 1u;
      const bool alone = (s_head[j / 32u] >> (j & 31u) & 1u) &&
                         (next == kTieSpan || (s_head[next / 32u] >> (next & 31u) & 1u));
      if (!alone) s_hi[j] = float_key(__ldg(hi + id[u]));
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kEach; ++u) {
      const uint32_t j = (uint32_t)u * 256u + threadIdx.x;
      if (j < kNearRun || j >= min(last, kNearRun + kTieTile)) continue;  // not of this tile
      // its run [a, b), as far as two words of heads on either side tell
      const uint32_t wi = j / 32u, upto = 0xffffffffu >> (31u - (j & 31u));
      const uint32_t h0 = s_head[wi] & upto, h1 = s_head[wi - 1u], h2 = s_head[wi - 2u];
      const uint32_t n0 = s_head[wi] & ~upto, n1 = s_head[wi + 1u], n2 = s_head[wi + 2u];
      const uint32_t base = wi * 32u, none = 2u * kTieSpan;
      const uint32_t a = h0 ? base + 31u - __clz(h0) : h1 ? base - 1u - __clz(h1) : h2 ? base - 33u - __clz(h2) : none;
      const uint32_t b = n0 ? base + __ffs(n0) - 1u : n1 ? base + 31u + __ffs(n1) : n2 ? base + 63u + __ffs(n2) : none;
      if (a != none && b != none && b - a <= kNearRun) {
        uint32_t at = t0 + a - kNearRun;
        if (b - a > 1u) {
          const uint32_t h = s_hi[j];
#pragma unroll 4
          for (uint32_t i = a; i < b; ++i) at += (s_hi[i] < h || (s_hi[i] == h && i < j)) ? 1u : 0u;
        }
        vals[at] = id[u];
      } else if (a == j) {
        const uint32_t i = t0 + j - kNearRun;
        const unsigned long long key = words[i] >> id_bits;
        // its end: equal at i + lo, not at i + up (or behind the set)
        uint32_t lo = kNearRun, up = 2u * kNearRun;
        while (up < n - i && (words[i + up] >> id_bits) == key) {
          lo = up;
          up *= 2u;
        }
        up = min(up, n - i);
        while (up - lo > 1u) {
          const uint32_t mid = lo + (up - lo) / 2u;
          if ((words[i + mid] >> id_bits) == key) lo = mid; else up = mid;
        }
        if (up <= kWarpRun)
          list[atomicAdd(&st->runs[0], 1u)] = make_uint2(i, up);
        else
          list[n / 2u - 1u - atomicAdd(&st->runs[1], 1u)] = make_uint2(i, up);
      }
    }
  }
}

// Largest cluster (CTAs) k_sort_cluster can run on the current device: 16
// (non-portable), else 8, else 0.
template <int ITEMS, bool PACKED>
int cluster_sort_ctas() {
  static std::atomic<int> best[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 0;
  }
  int b = best[dev].load(std::memory_order_relaxed);
  if (b == 0) {
    b = -1;
    const size_t smem = sizeof(ClusterSortSmem<ITEMS, PACKED>);
    if (cudaFuncSetAttribute(k_sort_cluster<ITEMS, PACKED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) == cudaSuccess &&
        cudaFuncSetAttribute(k_sort_cluster<ITEMS, PACKED>,
                             cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
      for (int c : {16, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(c);
        cfg.blockDim = dim3(kSmallThreads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, k_sort_cluster<ITEMS, PACKED>, &cfg) == cudaSuccess &&
            clusters > 0) {
          b = c;
          break;
        }
      }
    }
    cudaGetLastError();
    best[dev].store(b, std::memory_order_relaxed);
  }
  return b < 0 ? 0 : b;
}

// One cluster launch of k_sort_cluster if the set fits one cluster: *done =
// true then (or an error), else nothing is enqueued.
template <int ITEMS, bool PACKED>
cudaError_t try_sort_cluster(SortScratch sc, const SortSource& src, uint32_t n, int passes,
                             cudaStream_t s, bool* done) {
  *done = false;
  constexpr uint32_t kTile = kSmallThreads * ITEMS;
  const uint32_t ctas = (n + kTile - 1) / kTile;
  if (ctas > (uint32_t)cluster_sort_ctas<ITEMS, PACKED>()) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = sizeof(ClusterSortSmem<ITEMS, PACKED>);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const int out = PACKED ? 0 : passes & 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, k_sort_cluster<ITEMS, PACKED>, sc.keys[0], sc.vals[0],
                                     sc.keys[out], sc.vals[out], n, passes, src);
  if (e == cudaSuccess) {
    note_launches(1);
    *done = true;
  }
  return e;
}

// Co-resident CTAs of k_sort_grid on the current device, capped at
// kGridMaxTiles (0: not usable).
template <int ITEMS, bool PACKED>
int grid_sort_tiles(int sms) {
  static std::atomic<int> per_sm[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return 0;
  }
  int b = per_sm[dev].load(std::memory_order_relaxed);
  if (b == 0) {
    const size_t smem = sizeof(GridSortSmem<ITEMS, PACKED>);
    if (cudaFuncSetAttribute(k_sort_grid<ITEMS, PACKED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem) ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_sort_grid<ITEMS, PACKED>, kSmallThreads, smem)) {
      cudaGetLastError();
      b = 0;
    }
    per_sm[dev].store(b > 0 ? b : -1, std::memory_order_relaxed);
  }
  if (b < 0) return 0;
  return (int)std::min<long long>((long long)b * sms, kGridMaxTiles);
}

// One cooperative launch of k_sort_grid if the set fits its resident grid:
// *done = true then (or an error), else nothing is enqueued.
template <int ITEMS, bool PACKED>
cudaError_t try_sort_grid(SortScratch sc, const SortSource& src, uint32_t n, int passes,
                          Status* st, int sms, cudaStream_t s, bool* done) {
  *done = false;
  constexpr uint32_t kTile = kSmallThreads * ITEMS;
  const uint32_t tiles = (n + kTile - 1) / kTile;
  if (tiles > (uint32_t)grid_sort_tiles<ITEMS, PACKED>(sms)) return cudaSuccess;
  cudaError_t e;
  // both parities' group sums and the barrier counter start at zero
  uint32_t* sums = sc.lookback + kGridRowWords;
  if ((e = cudaMemsetAsync(sums, 0, sizeof(uint32_t) * (kGridSumWords + 1), s))) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles);
  cfg.blockDim = dim3(kSmallThreads);
  cfg.dynamicSmemBytes = sizeof(GridSortSmem<ITEMS, PACKED>);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, k_sort_grid<ITEMS, PACKED>, sc.keys[0], sc.vals[0], sc.keys[1], sc.vals[1],
                         n, passes, src, sc.lookback, sums + kGridSumWords, st);
  if (e == cudaErrorCooperativeLaunchTooLarge) {  // fewer SMs available than counted
    cudaGetLastError();
    return cudaSuccess;
  }
  if (e == cudaSuccess) {
    note_launches(1);
    *done = true;
  }
  return e;
}

}  // namespace

cudaError_t launch_debug_wait(const uint32_t* word, uint32_t limit, Status* st, cudaStream_t s) {
  k_debug_wait<<<1, 32, 0, s>>>(word, limit, st);
  note_launches(1);
  return cudaGetLastError();
}

size_t sort_lookback_words(uint32_t n) {
  const size_t tiles = ((size_t)n + kSortTile - 1) / kSortTile;
  // the onesweep look-back words, or the cooperative sort's rows, group sums and counter
  return std::max((size_t)kPasses * tiles * kRadix, kGridScratchWords);
}

namespace {

// The one-launch forms, smallest first: *done = false if none fits.
template <bool PACKED>
cudaError_t sort_in_one(SortScratch sc, const SortSource& src, uint32_t n, int passes,
                        Status* st, int sms, cudaStream_t s, bool* done) {
  // Up to 16 tiles of 2,048 keys: one cluster, keys kept on chip; else one
  // cooperative launch when every tile can be resident at once, with the
  // smallest tile that allows it.  Measured (8 passes, one GB300): 5,000
  // keys 33 us in a cluster, 53 cooperative, 51 in one CTA; 25,000 keys 41,
  // 57 (2,048-key tiles) and 100 (8,192-key tiles); 250,000 keys 76
  // cooperative.  Under stream capture too (the launches become graph nodes
  // with the same attributes): 256 batched instances in a graph took 187 us
  // with the multi-launch form recorded instead, 149 with these.
  cudaError_t e;
  if ((e = try_sort_cluster<4, PACKED>(sc, src, n, passes, s, done)) || *done) return e;
  if ((e = try_sort_grid<4, PACKED>(sc, src, n, passes, st, sms, s, done)) || *done) return e;
  if ((e = try_sort_grid<8, PACKED>(sc, src, n, passes, st, sms, s, done)) || *done) return e;
  return try_sort_grid<16, PACKED>(sc, src, n, passes, st, sms, s, done);
}

cudaError_t clear_onesweep(SortScratch sc, uint32_t tiles, int passes, cudaStream_t s) {
  cudaError_t e;
  if ((e = cudaMemsetAsync(sc.hist, 0, sizeof(uint32_t) * kPasses * kRadix, s))) return e;
  if ((e = cudaMemsetAsync(sc.counters, 0, sizeof(uint32_t) * kPasses, s))) return e;
  return cudaMemsetAsync(sc.lookback, 0, sizeof(uint32_t) * (size_t)passes * tiles * kRadix, s);
}

// Pass p; in the second half (the second key's passes, run first) its counts
// follow the first key's.
template <int FROM, bool LAST>
cudaError_t onesweep_packed_pass(SortScratch sc, const SortSource& src, uint32_t n, int p, int passes,
                                 bool second_half, Status* st, cudaStream_t s) {
  const uint32_t tiles = (n + kSortTile - 1) / kSortTile;
  const size_t smem = sizeof(PackedSmem);
  cudaError_t e = cudaFuncSetAttribute(k_onesweep_packed<FROM, LAST>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e) return e;
  const int at = second_half ? passes + p : p;
  k_onesweep_packed<FROM, LAST><<<tiles, kPackThreads, smem, s>>>(
      sc.keys[p & 1], src, sc.keys[(p & 1) ^ 1], sc.vals[0], n, src.id_bits + p * kRadixBits,
      sc.hist + at * kRadix, sc.lookback + (size_t)at * tiles * kRadix, sc.counters + at, second_half,
      !second_half && p + 1 == passes, st);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_tie_order(const unsigned long long* words, uint32_t n, int id_bits,
                             const float* hi, uint32_t* vals, uint2* list, Status* st, int sms,
                             cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t need = (n + kTieTile - 1) / kTieTile, cap = (uint32_t)sms * 16u;
  k_tie_order<<<need < cap ? need : cap, 256, 0, s>>>(words, n, id_bits, hi, vals, list, st);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sort_packed(SortScratch sc, const SortSource& src, uint32_t n, int key_bits,
                               Status* st, int sms, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const int passes = std::max((key_bits + kRadixBits - 1) / kRadixBits, 1);
  const int halves = src.both ? 2 : 1;
  cudaError_t e;
  bool done = false;
  if ((e = sort_in_one<true>(sc, src, n, passes, st, sms, s, &done)) || done) return e;
  const uint32_t tiles = (n + kSortTile - 1) / kSortTile;
  if ((e = clear_onesweep(sc, tiles, halves * passes, s))) return e;
  const uint32_t hb = std::min((n + kThreads * 16 - 1) / (kThreads * 16), (uint32_t)sms * 8u);
  if (src.both)
    k_histogram_packed<true><<<hb, kThreads, 0, s>>>(sc.keys[0], src, n, passes, sc.hist);
  else
    k_histogram_packed<false><<<hb, kThreads, 0, s>>>(sc.keys[0], src, n, passes, sc.hist);
  k_hist_scan<<<halves * passes, kRadix, 0, s>>>(sc.hist);
  if (src.both) {  // an even number of passes: the words return to keys[0]
    for (int p = 0; p < passes; ++p) {
      e = p == 0 ? onesweep_packed_pass<kFromSecond, false>(sc, src, n, p, passes, true, st, s)
                 : onesweep_packed_pass<kFromWords, false>(sc, src, n, p, passes, true, st, s);
      if (e) return e;
    }
  }
  for (int p = 0; p < passes; ++p) {
    const bool first = p == 0 && src.k32, last = p + 1 == passes && !src.words_out;
    e = first ? (last ? onesweep_packed_pass<kFromFirst, true>(sc, src, n, p, passes, false, st, s)
                      : onesweep_packed_pass<kFromFirst, false>(sc, src, n, p, passes, false, st, s))
              : (last ? onesweep_packed_pass<kFromWords, true>(sc, src, n, p, passes, false, st, s)
                      : onesweep_packed_pass<kFromWords, false>(sc, src, n, p, passes, false, st, s));
    if (e) return e;
  }
  note_launches(2u + (unsigned)(halves * passes));
  return cudaSuccess;
}

cudaError_t launch_sort64(SortScratch sc, uint32_t n, int passes, int* out_buf, Status* st, int sms,
                          cudaStream_t s) {
  *out_buf = 0;
  if (n <= 1 || passes <= 0) return cudaSuccess;
  if (passes > kPasses) passes = kPasses;
  cudaError_t e;
  bool done = false;
  if ((e = sort_in_one<false>(sc, SortSource{}, n, passes, st, sms, s, &done)) || done) {
    *out_buf = passes & 1;
    return e;
  }
  const uint32_t tiles = (n + kSortTile - 1) / kSortTile;
  if ((e = clear_onesweep(sc, tiles, passes, s))) return e;
  uint32_t hb = (n + kThreads * 16 - 1) / (kThreads * 16);
  if (hb > (uint32_t)sms * 4u) hb = (uint32_t)sms * 4u;
  k_histogram<<<hb, kThreads, 0, s>>>(sc.keys[0], n, sc.hist);
  k_hist_scan<<<kPasses, kRadix, 0, s>>>(sc.hist);
  const size_t smem = sizeof(OnesweepSmem);
  if ((e = cudaFuncSetAttribute(k_onesweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)smem)))
    return e;
  for (int p = 0; p < passes; ++p) {
    const int src = p & 1;
    k_onesweep<<<tiles, kThreads, smem, s>>>(sc.keys[src], sc.vals[src], sc.keys[src ^ 1],
                                             sc.vals[src ^ 1], n, p * kRadixBits,
                                             sc.hist + p * kRadix,
                                             sc.lookback + (size_t)p * tiles * kRadix,
                                             sc.counters + p, st);
  }
  note_launches(2u + (unsigned)passes);
  *out_buf = passes & 1;
  return cudaGetLastError();
}

}  // namespace ddm
