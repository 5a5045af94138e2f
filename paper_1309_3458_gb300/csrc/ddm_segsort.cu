// Re-sorts inside groups: the sort-tile-recursive refinement of an order.
//
// Dimension k >= 1 of a set is re-sorted by lower bound (the 24-bit locality
// key, stably) inside aligned groups of 2^g consecutive positions of each
// instance (a batched problem, a size class of the d >= 2 tree, or the whole
// update set).  A group is a contiguous range, and at the sizes that matter
// it fits one CTA's shared memory, so the re-sort needs no pass over the whole
// set: each CTA takes a chunk of whole groups (kSegTile positions, or 2^g if
// that is more), sorts it on chip and writes its ids back in place.
//
// This replaces a radix sort of (group, key) keys over the whole set -- two or
// three more digits for the group, and per digit either two grid barriers or a
// full read and write of keys and ids.  Bound by the ranking (instruction
// issue and shared-memory latency), not by memory: ids are read and written
// once and one coordinate per element is gathered.  Measured, whole calls: one
// match of 5e5 + 5e5 extents (d = 2) 425 -> 332 us, 4,096 batched instances
// (5.8e7 extents) 16.4 -> 13.8 ms, 256 of them in a CUDA graph 443 -> 299 us.
#include <algorithm>
#include <mutex>

#include "ddm_internal.cuh"

namespace ddm {
namespace {

constexpr int kRadix = 256;
constexpr int kPartWarps = 8;                      // warps whose counts a thread sums
constexpr int kKeyBits = 24;                       // locality key, see ddm_layout.cu

template <int THREADS, int ITEMS>
struct SegSmem {
  static constexpr int warps = THREADS / 32;
  static constexpr int parts = THREADS / kRadix;  // threads per digit
  static_assert(parts * kPartWarps == warps, "a thread per digit and eight warps");
  uint32_t whist[warps][kRadix];      // per-warp digit counts, then first slots within the digit
  uint32_t part[parts][kRadix];
  uint32_t total[kRadix];             // the tile's keys with each digit
  uint32_t first[kRadix];             // the digit's first slot in the tile
  uint32_t wtot[kRadix / 32];
  uint32_t base[kRadix];              // groups larger than a tile: running positions
  uint32_t range[2];                  // least and largest key of a chunk
  unsigned long long word[THREADS * ITEMS];
};

// Lanes of the warp holding the same 8-bit digit.
__device__ __forceinline__ uint32_t same_digit(uint32_t dig) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const uint32_t bit = (dig >> b) & 1u;
    const uint32_t votes = __ballot_sync(0xffffffffu, bit);
    peers &= bit ? votes : ~votes;
  }
  return peers;
}

// Stable ranking of one tile by one digit: item i of lane l in warp w is
// element w*32*ITEMS + i*32 + l.  Elements past `valid` hold the largest key,
// so they rank last; warps without a valid element skip the ranking.  The
// ballots of all items come first: only a read and a write of the warp's
// counters per item are left in the serial chain.
template <int THREADS, int ITEMS, typename Smem>
__device__ __forceinline__ void rank_digit(Smem& sm,
                                           const unsigned long long (&word)[ITEMS],
                                           uint32_t (&rank)[ITEMS], uint32_t valid, int shift) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t below = (1u << lane) - 1u;
  for (int t = lane; t < kRadix; t += 32) sm.whist[warp][t] = 0u;
  __syncwarp();
  if ((uint32_t)warp * (ITEMS * 32) < valid) {
    uint32_t peers[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) peers[i] = same_digit((uint32_t)(word[i] >> shift) & 255u);
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      uint32_t* h = &sm.whist[warp][(uint32_t)(word[i] >> shift) & 255u];
      const uint32_t before = *h;
      rank[i] = before + __popc(peers[i] & below);
      __syncwarp();
      if ((peers[i] & below) == 0u) *h = before + __popc(peers[i]);
      __syncwarp();
    }
  }
  __syncthreads();
  // Thread (part, digit): the digit's counts of a quarter of the warps ...
  const int dig = tid & (kRadix - 1), part = tid / kRadix;
  uint32_t c[kPartWarps], sum = 0;
#pragma unroll
  for (int j = 0; j < kPartWarps; ++j) {
    c[j] = sm.whist[part * kPartWarps + j][dig];
    sum += c[j];
  }
  sm.part[part][dig] = sum;
  __syncthreads();
  // ... become each warp's first slot within the digit, and the digits' totals
  // their first slots in the tile.
  uint32_t run = 0, all = 0;
#pragma unroll
  for (int q = 0; q < THREADS / kRadix; ++q) {
    const uint32_t v = sm.part[q][dig];
    run += q < part ? v : 0u;
    all += v;
  }
#pragma unroll
  for (int j = 0; j < kPartWarps; ++j) {
    sm.whist[part * kPartWarps + j][dig] = run;
    run += c[j];
  }
  uint32_t x = all;
  if (part == 0) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) sm.wtot[warp] = x;
    sm.total[dig] = all;
  }
  __syncthreads();
  if (part == 0) {
    uint32_t pre = 0;
    for (int q = 0; q < warp; ++q) pre += sm.wtot[q];
    sm.first[dig] = pre + x - all;
  }
  __syncthreads();
}

// One chunk of at most a tile.  Its words hold the key above the least key of
// the chunk, in as many bits as the range needs, with the group above that:
// coordinates of one scale range over some 20 of the 24 bits, so that a
// chunk of several groups usually takes three digits instead of four.  BITS: of
// the key; with all 32 the chunk is one group.
template <int THREADS, int ITEMS, int BITS, typename Smem>
__device__ __forceinline__ void sort_chunk(Smem& sm, uint32_t* vals, const float* lo_k,
                                           uint32_t len, int g) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool any = (uint32_t)warp * (ITEMS * 32) < len;  // warps past the chunk idle
  unsigned long long word[ITEMS];
  uint32_t rank[ITEMS];
  if (tid < 2) sm.range[tid] = tid ? 0u : 0xffffffffu;
  uint32_t id[ITEMS], key[ITEMS], least = 0xffffffffu, most = 0u;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t at = warp * (ITEMS * 32) + i * 32 + lane;
    id[i] = at < len ? vals[at] : 0u;
  }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t at = warp * (ITEMS * 32) + i * 32 + lane;
    if (at < len) {
      key[i] = float_key(__ldg(lo_k + id[i])) >> (32 - BITS);
      least = min(least, key[i]);
      most = max(most, key[i]);
    }
  }
  __syncthreads();
  if (any) {
    least = __reduce_min_sync(0xffffffffu, least);
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) {
      atomicMin(&sm.range[0], least);
      atomicMax(&sm.range[1], most);
    }
  }
  __syncthreads();
  least = sm.range[0];
  const int bits = 32 - __clz(sm.range[1] - least), groups = (int)((len - 1u) >> g);
  const int passes = max((bits + 32 - __clz(groups) + 7) / 8, 1);
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const uint32_t at = warp * (ITEMS * 32) + i * 32 + lane;
    uint32_t high = key[i] - least;
    if (BITS < 32) high |= (at >> g) << bits;
    word[i] = at < len ? ((unsigned long long)high << 32) | id[i] : ~0ull;
  }
  for (int p = 0; p < passes; ++p) {
    const int shift = 32 + 8 * p;
    rank_digit<THREADS, ITEMS>(sm, word, rank, len, shift);
    if (any) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const uint32_t d = (uint32_t)(word[i] >> shift) & 255u;
        sm.word[sm.first[d] + sm.whist[warp][d] + rank[i]] = word[i];
      }
    }
    __syncthreads();
    if (p + 1 < passes && any) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) word[i] = sm.word[warp * (ITEMS * 32) + i * 32 + lane];
    }
  }
  for (uint32_t q = tid; q < len; q += THREADS) vals[q] = (uint32_t)sm.word[q];
  __syncthreads();  // before the next chunk's words
}

// One group larger than a tile (an instance of millions of extents): the same
// digits, tile by tile through two scratch ranges in global memory.
template <int THREADS, int ITEMS, int BITS>
__device__ void sort_large_group(SegSmem<THREADS, ITEMS>& sm, uint32_t* vals, const float* lo_k,
                                 uint32_t len, unsigned long long* a, unsigned long long* b) {
  constexpr uint32_t kTile = THREADS * ITEMS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t q = tid; q < len; q += THREADS) {
    const uint32_t id = vals[q];
    a[q] = ((unsigned long long)(float_key(__ldg(lo_k + id)) >> (32 - BITS)) << 32) | id;
  }
  __syncthreads();
  for (int p = 0; p < BITS / 8; ++p) {
    const int shift = 32 + 8 * p;
    for (int t = tid; t < kRadix; t += THREADS) sm.base[t] = 0u;
    __syncthreads();
    for (uint32_t q = tid; q < len; q += THREADS)
      atomicAdd(&sm.base[(uint32_t)(__ldcg(a + q) >> shift) & 255u], 1u);
    __syncthreads();
    if (warp == 0) {  // exclusive scan of the 256 counts, eight per lane
      uint32_t c[8], sum = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        c[j] = sm.base[lane * 8 + j];
        sum += c[j];
      }
      uint32_t x = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      uint32_t run = x - sum;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        sm.base[lane * 8 + j] = run;
        run += c[j];
      }
    }
    __syncthreads();
    for (uint32_t t0 = 0; t0 < len; t0 += kTile) {
      const uint32_t valid = min(kTile, len - t0);
      unsigned long long word[ITEMS];
      uint32_t rank[ITEMS];
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const uint32_t at = warp * (ITEMS * 32) + i * 32 + lane;
        word[i] = at < valid ? __ldcg(a + t0 + at) : ~0ull;
      }
      rank_digit<THREADS, ITEMS>(sm, word, rank, valid, shift);
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const uint32_t at = warp * (ITEMS * 32) + i * 32 + lane;
        const uint32_t d = (uint32_t)(word[i] >> shift) & 255u;
        if (at < valid) b[sm.base[d] + sm.whist[warp][d] + rank[i]] = word[i];
      }
      __syncthreads();
      // padding words have digit 255 and come last: they do not count
      if (tid < kRadix) sm.base[tid] += sm.total[tid];
      __syncthreads();
    }
    unsigned long long* t = a;
    a = b;
    b = t;
  }
  for (uint32_t q = tid; q < len; q += THREADS) vals[q] = (uint32_t)__ldcg(a + q);
  __syncthreads();
}

// A chunk or group of `len` positions; a and b as sort_large_group.
template <int THREADS, int ITEMS, int BITS>
__device__ __forceinline__ void sort_range(SegSmem<THREADS, ITEMS>& sm, uint32_t* vals, const float* lo_k,
                                           uint32_t len, int g, unsigned long long* a,
                                           unsigned long long* b) {
  if (len > THREADS * ITEMS)
    sort_large_group<THREADS, ITEMS, BITS>(sm, vals, lo_k, len, a, b);
  else if (len > THREADS * 2 || (ITEMS == 2 && len > THREADS))
    sort_chunk<THREADS, ITEMS, BITS>(sm, vals, lo_k, len, g);
  else if (len > THREADS)
    sort_chunk<THREADS, 2, BITS>(sm, vals, lo_k, len, g);
  else if (len > 1)
    sort_chunk<THREADS, 1, BITS>(sm, vals, lo_k, len, g);
}

// Re-sort of one set.  With `off` null: one instance of `total` positions and
// group exponent g_one; else instance i owns positions [off[i], off[i+1]) with
// exponent glog2[i] (0: left as it is) and chunks [cbase[i], cbase[i+1]).
template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
k_segsort(uint32_t* __restrict__ vals, const float* __restrict__ lo_k, uint32_t total, int g_one,
          const unsigned long long* __restrict__ off, const int* __restrict__ glog2,
          const unsigned long long* __restrict__ cbase, uint32_t count,
          unsigned long long* __restrict__ tmp0, unsigned long long* __restrict__ tmp1) {
  constexpr uint32_t kTile = THREADS * ITEMS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SegSmem<THREADS, ITEMS>& sm = *reinterpret_cast<SegSmem<THREADS, ITEMS>*>(smem_raw);
  const unsigned long long chunks = off ? cbase[count] : ((unsigned long long)total + kTile - 1) / kTile;
  for (unsigned long long c = blockIdx.x; c < chunks; c += gridDim.x) {
    unsigned long long begin = c * kTile, end = min(begin + kTile, (unsigned long long)total);
    int g = g_one;
    if (off) {
      const uint32_t b = warp_owner(cbase, count, c);  // the instance whose chunks include c
      g = glog2[b];
      const unsigned long long size = max((unsigned long long)kTile, 1ull << g);
      begin = off[b] + (c - cbase[b]) * size;
      end = min(begin + size, off[b + 1]);
    }
    const uint32_t len = (uint32_t)(end - begin);
    sort_range<THREADS, ITEMS, kKeyBits>(sm, vals + begin, lo_k, len, g, tmp0 + begin, tmp1 + begin);
  }
}

// The runs of equal lower bounds that k_tie_order has listed: ids of each in
// the order of their upper bound (stably).  A warp counts, for every element of
// its run, those before it; a CTA sorts its run like a chunk of a re-sort, by
// all 32 bits.  Small CTAs: while the updates are sorted on another stream,
// larger ones would wait for a whole SM to fall idle (a match of 2.5e7 + 2.5e7
// extents 6.10 -> 6.47 ms with CTAs of 1,024 threads).
constexpr int kTieThreads = 256, kTieItems = 8;
static_assert(kTieThreads * kTieItems == (int)kCtaRun, "runs of a CTA are sorted on chip");

// A run of at most kWarpRun elements by one warp (a run of 200 took it 40 us).
__device__ __forceinline__ void warp_run(const unsigned long long* __restrict__ words, uint2 run,
                                         unsigned long long idm, const float* __restrict__ hi,
                                         uint32_t* __restrict__ vals) {
  constexpr int EACH = (int)kWarpRun / 32;
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t id[EACH], key[EACH], rank[EACH];
#pragma unroll
  for (int c = 0; c < EACH; ++c) {
    const uint32_t at = c * 32u + lane;
    id[c] = at < run.y ? (uint32_t)(words[run.x + at] & idm) : 0u;
    rank[c] = 0u;
  }
#pragma unroll
  for (int c = 0; c < EACH; ++c)
    key[c] = c * 32u + lane < run.y ? float_key(__ldg(hi + id[c])) : 0xffffffffu;
#pragma unroll
  for (int c2 = 0; c2 < EACH; ++c2) {
    if (c2 * 32u >= run.y) break;  // warp-uniform
#pragma unroll 4
    for (uint32_t l = 0; l < 32u; ++l) {
      const uint32_t k2 = __shfl_sync(0xffffffffu, key[c2], l);
#pragma unroll
      for (int c = 0; c < EACH; ++c)
        rank[c] += (k2 < key[c] || (k2 == key[c] && c2 * 32u + l < c * 32u + lane)) ? 1u : 0u;
    }
  }
#pragma unroll
  for (int c = 0; c < EACH; ++c)
    if (c * 32u + lane < run.y) vals[run.x + rank[c]] = id[c];
}

__global__ void __launch_bounds__(kTieThreads, 4)
k_long_ties(unsigned long long* __restrict__ words, uint32_t n, int id_bits,
            const float* __restrict__ hi, uint32_t* __restrict__ vals, const uint2* __restrict__ list,
            unsigned long long* __restrict__ tmp, const Status* __restrict__ st) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto& sm = *reinterpret_cast<SegSmem<kTieThreads, kTieItems>*>(smem_raw);
  const uint32_t short_runs = st->runs[0], long_runs = st->runs[1];
  const unsigned long long idm = (1ull << id_bits) - 1ull;
  for (uint32_t e = blockIdx.x * (kTieThreads / 32) + threadIdx.x / 32u; e < short_runs;
       e += gridDim.x * (kTieThreads / 32)) {
    warp_run(words, list[e], idm, hi, vals);
  }
  for (uint32_t e = blockIdx.x; e < long_runs; e += gridDim.x) {
    const uint2 run = list[n / 2u - 1u - e];
    for (uint32_t q = threadIdx.x; q < run.y; q += kTieThreads)
      vals[run.x + q] = (uint32_t)(words[run.x + q] & idm);
    __syncthreads();
    sort_range<kTieThreads, kTieItems, 32>(sm, vals + run.x, hi, run.y, 31, words + run.x, tmp + run.x);
  }
}

// Thresholds of the group exponents: entry (d * 8 + k) * 32 + g = the least
// leaf count nb at which str_group_log2's G = 32 * nb^((d-k)/d) rounds to 2^g
// or more (unclamped, without shift).  The double-precision pow and log2 of
// the rule cost a launch of one small kernel 7 us per dimension; comparing
// with thresholds gives the same exponents (G grows by far more than a
// rounding error from one nb to the next).
__device__ __forceinline__ int group_exponent(double nb, int d, int k) {
  return (int)floor(log2(32.0 * pow(nb, (double)(d - k) / (double)d)) + 0.5);
}
static __device__ uint32_t g_group_table[(DDM_MAX_DIMS + 1) * 8 * 32];

__global__ void k_group_table() {
  const int d = blockIdx.x / 8, k = blockIdx.x % 8, g = threadIdx.x;
  if (d < 2 || k < 1 || k >= d) return;
  uint32_t lo = 1, hi = 1u << 26;  // more than 2^30 / 32 leaves
  while (lo < hi) {
    const uint32_t mid = (lo + hi) / 2;
    if (group_exponent((double)mid, d, k) >= g) hi = mid; else lo = mid + 1;
  }
  g_group_table[(d * 8 + k) * 32 + g] = lo;
}

// str_group_log2 by the table.
__device__ __forceinline__ int table_group(uint32_t n, int d, int k, int shift) {
  if (n < 64u) return 0;
  const uint32_t nb = (n + 31u) / 32u;
  const uint32_t* t = g_group_table + (d * 8 + k) * 32;
  int lo = 0, hi = 32;  // t[lo] <= nb (G >= 32 for every nb), t[hi] > nb
  while (hi - lo > 1) {
    const int mid = (lo + hi) / 2;
    if (t[mid] <= nb) lo = mid; else hi = mid;
  }
  const int g = lo + shift;
  if (g < 6 || (1ull << g) >= (unsigned long long)n) return 0;
  return g;
}
// The exponent used for dimension k: strictly smaller than those before it.
__device__ __forceinline__ int used_group(uint32_t n, int d, int k, int shift) {
  int g = table_group(n, d, k, shift);
  for (int j = 1; j < k && g > 0; ++j) {
    const int gp = table_group(n, d, j, shift);
    if (gp > 0 && g >= gp) g = 0;
  }
  return g;
}
__device__ __forceinline__ uint32_t chunks_of(uint32_t n, int g, uint32_t tile) {
  if (g == 0) return 0u;
  const unsigned long long size = max((unsigned long long)tile, 1ull << g);
  return (uint32_t)((n + size - 1) / size);
}

// Exclusive scan of one value per thread over 1,024 threads; *total = the sum.
__device__ __forceinline__ uint32_t scan1024(uint32_t v, uint32_t* s_w, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  uint32_t w = s_w[lane];  // every warp scans the 32 warp totals
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
    if (lane >= o) w += y;
  }
  *total = __shfl_sync(0xffffffffu, w, 31);
  const uint32_t pre = __shfl_sync(0xffffffffu, w, (warp + 31) & 31);
  __syncthreads();
  return (warp ? pre : 0u) + x - v;
}

// Sum of one value per thread over 1,024 threads.
__device__ __forceinline__ unsigned long long sum1024(unsigned long long v, unsigned long long* s_w) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) s_w[threadIdx.x >> 5] = v;
  __syncthreads();
  v = s_w[lane];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  return v;
}

// Batched sets: the prefix of leaves of a padded tree and, for every dimension
// k >= 1, each instance's group exponent and the prefix of chunks.  A CTA takes
// kPlanTile instances.  Up to that many are one launch, where a launch per step
// (counts, scan) put seven on the way of a small batch; more take two, the
// first for the tiles' sums ([0]: leaves, [k]: chunks, [d]: whether the
// offsets are unsound), of which each CTA of the second adds up those before it:
// a match of a million instances, all but one empty, took 1,170 us with one
// CTA, 211 now.  Offsets that descend or pass the set's `total` get no chunks:
// the re-sorts move ids in place, and chunks of such offsets could overlap or
// lie outside the set.
constexpr uint32_t kPlanEach = 4, kPlanTile = 1024 * kPlanEach;
enum { kPlanOne, kPlanSums, kPlanRest };  // one tile; the two launches of several
template <int PHASE>
__global__ void __launch_bounds__(1024, 1)
k_batch_plan(const unsigned long long* __restrict__ off, uint32_t count, uint32_t total, int d,
             int shift, uint32_t tile, int* __restrict__ glog2, unsigned long long* __restrict__ cbase,
             unsigned long long* __restrict__ leaf_off, unsigned long long* __restrict__ sums) {
  __shared__ unsigned long long s_sum[PHASE == kPlanOne ? 1 : 32];
  __shared__ uint32_t s_w[32];
  const uint32_t tiles = gridDim.x, me = blockIdx.x;
  const uint32_t i0 = me * kPlanTile + threadIdx.x * kPlanEach;
  bool bad = false;
  uint32_t n[kPlanEach];
#pragma unroll
  for (int u = 0; u < (int)kPlanEach; ++u) {
    n[u] = 0u;
    if (i0 + u < count) {
      const unsigned long long a = off[i0 + u], b = off[i0 + u + 1];
      bad |= b < a || b > total;
      n[u] = (uint32_t)(b - a);
    }
  }
#pragma unroll
  for (int k = 0; k < DDM_MAX_DIMS; ++k) {
    if (k >= d || (k == 0 && !leaf_off)) continue;
    uint32_t v[kPlanEach], sum = 0, all;
#pragma unroll
    for (int u = 0; u < (int)kPlanEach; ++u) {
      if (k == 0) {
        v[u] = (n[u] + 31u) / 32u;
      } else {
        const int g = used_group(n[u], d, k, shift);
        if (PHASE != kPlanSums && i0 + u < count) glog2[(size_t)k * count + i0 + u] = g;
        v[u] = chunks_of(n[u], g, tile);
      }
      sum += v[u];
    }
    if (PHASE == kPlanSums) {
      const unsigned long long mine = sum1024(sum, s_sum);
      if (threadIdx.x == 0) sums[(size_t)k * tiles + me] = mine;
      continue;
    }
    unsigned long long before = 0;
    if (PHASE == kPlanRest) {
      for (uint32_t t = threadIdx.x; t < me; t += 1024u) before += sums[(size_t)k * tiles + t];
      before = sum1024(before, s_sum);
    }
    unsigned long long at = before + scan1024(sum, s_w, &all);
    unsigned long long* out = k == 0 ? leaf_off : cbase + (size_t)k * (count + 1u);
#pragma unroll
    for (int u = 0; u < (int)kPlanEach; ++u) {
      if (i0 + u < count) out[i0 + u] = at;
      at += v[u];
    }
    if (me + 1u == tiles && threadIdx.x == 0) out[count] = before + all;
  }
  if (PHASE == kPlanRest && me + 1u == tiles)
    for (uint32_t t = threadIdx.x; t < me; t += 1024u) bad |= sums[(size_t)d * tiles + t] != 0ull;
  bad = __syncthreads_or(bad);
  if (threadIdx.x != 0) return;
  if (PHASE == kPlanSums) {
    sums[(size_t)d * tiles + me] = bad;
  } else if (bad && me + 1u == tiles) {
    for (int k = 1; k < d; ++k) cbase[(size_t)k * (count + 1u) + count] = 0ull;
  }
}

// Exclusive scan of 256 values over the CTA's 256 threads; *total = their sum.
__device__ __forceinline__ uint32_t scan256(uint32_t v, uint32_t* s_w, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  uint32_t pre = 0, all = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    pre += q < warp ? s_w[q] : 0u;
    all += s_w[q];
  }
  __syncthreads();
  *total = all;
  return pre + x - v;
}

// Size classes (one CTA): offsets of the 256 classes from their histogram, and
// for every dimension k >= 1 their group exponents and chunk prefixes.
__global__ void __launch_bounds__(256)
k_class_plan(const uint32_t* __restrict__ hist, int d,
             int shift, ClassPlan plan) {
  __shared__ uint32_t s_w[8];
  const int i = threadIdx.x;
  const uint32_t n = hist[i];
  uint32_t total;
  const uint32_t at = scan256(n, s_w, &total);
  plan.off[i] = at;
  if (i == 255) plan.off[256] = total;
  for (int k = 1; k < d; ++k) {
    const int g = used_group(n, d, k, shift);
    const uint32_t c = chunks_of(n, g, plan.tile[k]);
    const uint32_t first = scan256(c, s_w, &total);
    plan.glog2[k * 256 + i] = g;
    plan.cbase[k * 257 + i] = first;
    if (i == 255) plan.cbase[k * 257 + 256] = total;
  }
}

template <int THREADS, int ITEMS>
cudaError_t launch_segsort_items(uint32_t* vals, const float* lo_k, uint32_t total, int g,
                                 const SegPlan& plan, unsigned long long* tmp0,
                                 unsigned long long* tmp1, int sms, cudaStream_t s) {
  const size_t smem = sizeof(SegSmem<THREADS, ITEMS>);
  cudaError_t e = cudaFuncSetAttribute(k_segsort<THREADS, ITEMS>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e) return e;
  // at most one chunk per instance beyond the whole tiles
  const uint64_t most = (uint64_t)total / (THREADS * ITEMS) + (plan.off ? plan.count : 0u) + 1u;
  const uint32_t blocks = (uint32_t)std::min<uint64_t>(most, (uint64_t)sms * (2048 / THREADS));
  k_segsort<THREADS, ITEMS><<<blocks, THREADS, smem, s>>>(vals, lo_k, total, g, plan.off, plan.glog2,
                                                     plan.cbase, plan.count, tmp0, tmp1);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// Fills the current device's table, once per process: on a stream of its own,
// so that no other stream's work is waited for.
cudaError_t ready_group_table() {
  static std::mutex lock;
  static bool done[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e) return e;
  std::lock_guard<std::mutex> hold(lock);
  if (dev >= 0 && dev < 64 && done[dev]) return cudaSuccess;
  cudaStream_t s = nullptr;
  if ((e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking))) return e;
  k_group_table<<<(DDM_MAX_DIMS + 1) * 8, 32, 0, s>>>();
  note_launches(1);
  e = cudaGetLastError();
  if (!e) e = cudaStreamSynchronize(s);
  cudaStreamDestroy(s);
  if (!e && dev >= 0 && dev < 64) done[dev] = true;
  return e;
}

size_t batch_plan_words(uint32_t count, int d) {
  const uint32_t tiles = (count + kPlanTile - 1u) / kPlanTile;
  return tiles > 1u ? (size_t)tiles * (d + 1) : 0u;
}

cudaError_t launch_batch_plan(const unsigned long long* off, uint32_t count, uint32_t total, int d,
                              int shift, int tile_log2, int* glog2, unsigned long long* cbase,
                              unsigned long long* leaf_off, unsigned long long* sums,
                              cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const uint32_t tiles = (count + kPlanTile - 1u) / kPlanTile, tile = 1u << tile_log2;
#define DDM_PLAN(PHASE)                                                                           \
  k_batch_plan<PHASE><<<tiles, 1024, 0, s>>>(off, count, total, d, shift, tile, glog2, cbase, leaf_off, sums)
  if (tiles == 1u) {
    DDM_PLAN(kPlanOne);
  } else {
    DDM_PLAN(kPlanSums);
    DDM_PLAN(kPlanRest);
  }
#undef DDM_PLAN
  note_launches(tiles > 1u ? 2u : 1u);
  return cudaGetLastError();
}

cudaError_t launch_class_plan(const uint32_t* hist, int d, int shift, const ClassPlan& plan,
                              cudaStream_t s) {
  k_class_plan<<<1, 256, 0, s>>>(hist, d, shift, plan);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_long_ties(unsigned long long* words, uint32_t n, int id_bits, const float* hi,
                             uint32_t* vals, const uint2* list, unsigned long long* tmp,
                             const Status* st, int sms, cudaStream_t s) {
  if (n <= 1) return cudaSuccess;
  const size_t smem = sizeof(SegSmem<kTieThreads, kTieItems>);
  cudaError_t e = cudaFuncSetAttribute(k_long_ties, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e) return e;
  k_long_ties<<<(uint32_t)sms * 4u, kTieThreads, smem, s>>>(words, n, id_bits, hi, vals, list, tmp, st);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_segsort(uint32_t* vals, const float* lo_k, uint32_t total, int g,
                           const SegPlan& plan, int tile_log2, unsigned long long* tmp0,
                           unsigned long long* tmp1, int sms, cudaStream_t s) {
  if (total <= 1) return cudaSuccess;
  if (tile_log2 == kSegTileLog2Max)
    return launch_segsort_items<1024, 8>(vals, lo_k, total, g, plan, tmp0, tmp1, sms, s);
  if (tile_log2 == 10)
    return launch_segsort_items<1024, 1>(vals, lo_k, total, g, plan, tmp0, tmp1, sms, s);
  if (tile_log2 == 11)
    return launch_segsort_items<1024, 2>(vals, lo_k, total, g, plan, tmp0, tmp1, sms, s);
  // More chunks than SMs: CTAs of half the threads, two to an SM, so that one
  // ranks while the other waits (2 x 2.9e7 positions of 4,096 instances: 2.00
  // ms with CTAs of 1,024 threads and all 24 key bits, 1.34 now).  Else a
  // chunk's latency counts: more threads.
  if ((total >> kSegTileLog2) > (uint32_t)sms)
    return launch_segsort_items<512, 8>(vals, lo_k, total, g, plan, tmp0, tmp1, sms, s);
  return launch_segsort_items<1024, 4>(vals, lo_k, total, g, plan, tmp0, tmp1, sms, s);
}

}  // namespace ddm
