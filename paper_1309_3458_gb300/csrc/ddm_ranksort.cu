// First order of a small set in one launch: validation, sort keys and a sort
// by counting.
//
// The rank of an extent is the number of extents with a smaller key (or an
// equal one and a smaller id): n^2 comparisons, spread over the whole chip,
// with no passes and no barriers between CTAs.  For a few thousand extents
// that is less work than waiting: the cluster radix sort's eight passes of
// 5,000 keys take 33 us of barriers and rankings behind a separate validation
// launch.  Bound by the integer compares (half rate on the ALU pipe; about 20
// 64-bit compares per clock and SM measured).  Quadratic, so only for small
// sets (rank_sort_max); the order is exactly the stable radix sort's.  One
// match of 5,000 + 5,000 extents: 107 -> 86 us.
#include "ddm_internal.cuh"

namespace ddm {
namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr uint32_t kChunk = 2048;  // keys staged at a time
constexpr uint32_t kOwn = 64;      // extents ranked by a CTA

// Sort keys as in ddm_layout.cu: kTree (lo, hi) of dimension 0 in 64 bits;
// kLocal the top 24 bits of lo; kClass those below the size class.
template <int MODE>
struct KeyOf {
  using type = uint32_t;
};
template <>
struct KeyOf<kRankTree> {
  using type = unsigned long long;
};

template <int MODE>
__device__ __forceinline__ typename KeyOf<MODE>::type key_of(int d, const float* __restrict__ lo,
                                                             const float* __restrict__ hi,
                                                             uint32_t n, uint32_t i) {
  const float a = __ldg(lo + i);
  if constexpr (MODE == kRankTree) {
    return ((unsigned long long)float_key(a) << 32) | float_key(__ldg(hi + i));
  } else {
    uint32_t key = float_key(a) >> 8;
    if constexpr (MODE == kRankClass) {
      float side = 0.0f;
      for (int k = 0; k < d; ++k)
        side = fmaxf(side, __ldg(hi + (size_t)k * n + i) - __ldg(lo + (size_t)k * n + i));
      key |= ((__float_as_uint(side) >> 23) & 0xffu) << 24;
    }
    return key;
  }
}

// Four keys with one shared-memory load (two for 64-bit keys).
__device__ __forceinline__ void load4(uint32_t (&k)[4], const uint32_t* p) {
  const uint4 v = *reinterpret_cast<const uint4*>(p);
  k[0] = v.x;
  k[1] = v.y;
  k[2] = v.z;
  k[3] = v.w;
}
__device__ __forceinline__ void load4(unsigned long long (&k)[4], const unsigned long long* p) {
  const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p);
  const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(p + 2);
  k[0] = a.x;
  k[1] = a.y;
  k[2] = b.x;
  k[3] = b.y;
}

// A CTA ranks 64 extents, two per lane; its warps share the comparisons.
// Every key loaded (a broadcast of four) serves both: with one extent per
// lane and one key per load the loads bound it, at a third of the rate.
template <int MODE>
__global__ void __launch_bounds__(kThreads)
k_rank_sort(int d, const float* __restrict__ lo, const float* __restrict__ hi, uint32_t n,
            uint32_t* __restrict__ vals, uint32_t* __restrict__ hist, float2* __restrict__ aos,
            float2* __restrict__ qe, uint32_t* __restrict__ qid, Status* __restrict__ st) {
  using Key = typename KeyOf<MODE>::type;
  __shared__ __align__(16) Key s_key[kChunk];
  __shared__ uint32_t s_rank[kWarps][kOwn];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t i0 = blockIdx.x * kOwn, ia = i0 + lane, ib = ia + 32u;
  const Key mine_a = ia < n ? key_of<MODE>(d, lo, hi, n, ia) : Key(0);
  const Key mine_b = ib < n ? key_of<MODE>(d, lo, hi, n, ib) : Key(0);
  uint32_t ra = 0, rb = 0;
  for (uint32_t c0 = 0; c0 < n; c0 += kChunk) {
    const uint32_t len = min(kChunk, n - c0), len4 = (len + 3u) & ~3u;
    if (c0) __syncthreads();
    for (uint32_t j = threadIdx.x; j < len4; j += kThreads)
      s_key[j] = j < len ? key_of<MODE>(d, lo, hi, n, c0 + j) : ~Key(0);  // padding: below nothing
    __syncthreads();
    // Warp w compares with the chunk's keys [a, b), whole fours: those before
    // the CTA's own extents count when equal too, those after them do not.
    const uint32_t per = kChunk / kWarps, a = min(warp * per, len4), b = min(a + per, len4);
    const uint32_t m0 = min(max(i0, c0 + a), c0 + b) - c0;
    const uint32_t m1 = min(max(i0 + kOwn, c0 + a), c0 + b) - c0;
    Key k[4];
#pragma unroll 4
    for (uint32_t j = a; j < m0; j += 4u) {
      load4(k, &s_key[j]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ra += k[u] <= mine_a ? 1u : 0u;
        rb += k[u] <= mine_b ? 1u : 0u;
      }
    }
    for (uint32_t j = m0; j < m1; ++j) {
      const Key kj = s_key[j];
      const uint32_t g = c0 + j;
      ra += (kj < mine_a || (kj == mine_a && g < ia)) ? 1u : 0u;
      rb += (kj < mine_b || (kj == mine_b && g < ib)) ? 1u : 0u;
    }
#pragma unroll 4
    for (uint32_t j = m1; j < b; j += 4u) {
      load4(k, &s_key[j]);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ra += k[u] < mine_a ? 1u : 0u;
        rb += k[u] < mine_b ? 1u : 0u;
      }
    }
  }
  s_rank[warp][lane] = ra;
  s_rank[warp][lane + 32] = rb;
  __syncthreads();
  if (threadIdx.x >= kOwn) return;
  const uint32_t i = i0 + threadIdx.x;
  const bool valid = i < n;
  const Key mine = warp ? mine_b : mine_a;  // threads 32..63 finish the second half
  uint32_t rank = 0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) rank += s_rank[w][threadIdx.x];
  bool bad = false;
  if (valid && DDM_IN_BOUNDS(rank < n, st)) {
    vals[rank] = i;
    for (int k = 0; k < d; ++k) {
      const float a = __ldg(lo + (size_t)k * n + i), b = __ldg(hi + (size_t)k * n + i);
      bad |= !(a <= b);  // false for NaN as well as for lo > hi
      if (aos) aos[(size_t)i * d + k] = make_float2(a, b);
      if (qe) qe[(size_t)k * n + rank] = make_float2(a, b);
    }
    if (qid) qid[rank] = i;
    if constexpr (MODE == kRankClass) atomicAdd(&hist[(uint32_t)mine >> 24], 1u);
  }
  if (__ballot_sync(0xffffffffu, bad) && lane == 0) atomicOr(&st->err, kErrExtent);
}

}  // namespace

cudaError_t launch_rank_sort(int mode, int d, const float* lo, const float* hi, uint32_t n,
                             uint32_t* vals, uint32_t* hist, float2* aos, float2* qe, uint32_t* qid,
                             Status* st, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint32_t blocks = (n + kOwn - 1u) / kOwn;
  switch (mode) {
    case kRankTree:
      k_rank_sort<kRankTree><<<blocks, kThreads, 0, s>>>(d, lo, hi, n, vals, hist, aos, qe, qid, st);
      break;
    case kRankLocal:
      k_rank_sort<kRankLocal><<<blocks, kThreads, 0, s>>>(d, lo, hi, n, vals, hist, aos, qe, qid, st);
      break;
    case kRankClass:
      k_rank_sort<kRankClass><<<blocks, kThreads, 0, s>>>(d, lo, hi, n, vals, hist, aos, qe, qid, st);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace ddm
