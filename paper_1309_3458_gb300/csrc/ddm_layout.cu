// Input validation, sort keys and gathers of the structure-of-arrays layout.
//
// Every extent must have lo <= hi with no NaN in every dimension (the
// paper's segments [low, high], Section III-A); a violation raises
// kErrExtent.  For the subscription set of a d = 1 tree the same pass emits
// the lower bound's key; ties are put in the order of their upper bounds
// after the sort (ddm_sort.cu), or, if one value abounds, the set is sorted
// by both bounds: the interval tree order of Section IV, with
// remaining ties in id order.  Every other order (d > 1 trees, the updates) is a locality order:
// its keys hold the top 24 bits of key(lo) below a class, group or instance.
//
// For d > 1 the order is then refined one dimension at a time: inside
// aligned groups of consecutive positions the extents are re-sorted by their
// lower bound in the next dimension (on chip, ddm_segsort.cu; groups too
// large for that through k_rekey's (group, key(lo_k)) keys).  Each group stays a contiguous range of the dimension-0 order, so
// the top of the tree still follows the paper's lower-bound order, while the
// small subtrees near the leaves become compact in every dimension.  For the
// tree with d > 1 the subscriptions are first grouped by size class
// (k_validate_class: class, then lower bound), and every class is refined
// with groups sized for it, like the instances of a batched set.
#include "ddm_internal.cuh"

namespace ddm {
namespace {

constexpr int kThreads = 256;
// Locality keys (every sort but the d = 1 tree's): the top 24 bits of the
// order-preserving float key -- sign, exponent and 15 mantissa bits, about
// 3e-5 relative -- below a group / class / instance number.  Such an order
// is a heuristic (any order gives the same pairs), and dropping the low
// byte saves one radix pass per sort.
constexpr int kLocalityBits = 24;
constexpr int kLocalityDrop = 32 - kLocalityBits;

// Whether one value of the lower bound abounds in a set (d = 1 tree): one CTA
// samples kSample of the bounds and counts the most frequent.  From four of a
// kind, and more than kCtaRun + cnt / 512 of the set by that share, the set is
// sorted by both bounds; fewer are put in order in place, a run at a time
// (ddm_sort.cu): a CTA takes 22 us per 2,048 of a run beyond that, four more
// digits some 20 us and 20 per million.  Builds of
// 5e5 extents, always by both bounds and now: distinct bounds 139 and 119 us, 12,500
// values 139 and 130, 500 values 137 and 144, one value 138 and 145, 1% at one
// value 139 and 149 (195 when such a run had the whole set sorted once more).
constexpr int kSample = 1024;
__device__ void sample_ties(const float* __restrict__ lo, uint32_t cnt, Status* __restrict__ st) {
  constexpr uint32_t kSlots = 2 * kSample, kEmpty = 0xffffffffu;
  __shared__ uint32_t s_key[kSlots], s_cnt[kSlots];
  __shared__ uint32_t s_most;
  for (uint32_t j = threadIdx.x; j < kSlots; j += kThreads) {
    s_key[j] = kEmpty;
    s_cnt[j] = 0u;
  }
  if (threadIdx.x == 0) s_most = 0u;
  uint32_t key[kSample / kThreads];
#pragma unroll
  for (int u = 0; u < kSample / kThreads; ++u) {
    const uint32_t j = (uint32_t)u * kThreads + threadIdx.x;
    key[u] = float_key(__ldg(lo + (uint32_t)((unsigned long long)j * cnt / kSample)));
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kSample / kThreads; ++u) {  // never kEmpty but for NaN
    uint32_t at = (key[u] * 2654435761u) >> 21;   // 11 bits
    for (uint32_t tries = 0; tries < 16u; ++tries, at = (at + 1u) & (kSlots - 1u)) {
      const uint32_t was = atomicCAS(&s_key[at], kEmpty, key[u]);
      if (was != key[u] && was != kEmpty) continue;
      atomicAdd(&s_cnt[at], 1u);
      break;
    }
  }
  __syncthreads();
  uint32_t most = 0;
  for (uint32_t j = threadIdx.x; j < kSlots; j += kThreads) most = max(most, s_cnt[j]);
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0) atomicMax(&s_most, most);
  __syncthreads();
  if (threadIdx.x != 0) return;
  st->both = s_most >= 4u && (unsigned long long)s_most * cnt / kSample > kCtaRun + cnt / 512u;
  st->runs[0] = st->runs[1] = 0u;
}

// TREE: the d = 1 tree's keys (whole), else a locality order's.
template <bool TREE>
__global__ void __launch_bounds__(kThreads)
k_validate(int d, const float* __restrict__ lo, const float* __restrict__ hi, uint32_t cnt,
           uint32_t* __restrict__ k32, float2* __restrict__ aos, Status* __restrict__ st) {
  bool bad = false;
  uint32_t blocks = gridDim.x;
  if constexpr (TREE) {  // the last CTA looks for ties
    if (blockIdx.x == --blocks) {
      sample_ties(lo, cnt, st);
      return;
    }
  }
  const uint32_t stride = blocks * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    // Row loads are coalesced: consecutive lanes read consecutive floats.
    for (int k = 0; k < d; ++k) {
      const float a = __ldg(lo + (size_t)k * cnt + i);
      const float b = __ldg(hi + (size_t)k * cnt + i);
      bad |= !(a <= b);  // false for NaN as well as for lo > hi
      if (aos) aos[(size_t)i * d + k] = make_float2(a, b);
    }
    if (k32) k32[i] = float_key(__ldg(lo + i)) >> (TREE ? 0 : kLocalityDrop);
  }
  if (__ballot_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&st->err, kErrExtent);
}

__global__ void __launch_bounds__(kThreads)
k_rekey(const uint32_t* __restrict__ vals, const float* __restrict__ lo_k, uint32_t cnt, int glog2,
        unsigned long long* __restrict__ keys, int id_bits) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    const uint32_t id = vals[i];
    const unsigned long long k = ((unsigned long long)(i >> glog2) << kLocalityBits) |
                                 (float_key(__ldg(lo_k + id)) >> kLocalityDrop);
    keys[i] = id_bits ? (k << id_bits) | id : k;
  }
}

__global__ void __launch_bounds__(kThreads)
k_gather(int d, const uint32_t* __restrict__ vals, const float* __restrict__ lo,
         const float* __restrict__ hi, const float2* __restrict__ aos, uint32_t cnt,
         float2* __restrict__ qe, uint32_t* __restrict__ qid) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    const uint32_t id = vals[i];
    qid[i] = id;
    for (int k = 0; k < d; ++k)
      qe[(size_t)k * cnt + i] = aos ? aos[(size_t)id * d + k]
                                    : make_float2(__ldg(lo + (size_t)k * cnt + id),
                                                  __ldg(hi + (size_t)k * cnt + id));
  }
}

// Validation plus the first sort key of the tree order for d >= 2: the size
// class of the extent -- the binary exponent of its largest side (the float
// exponent field) -- above the top 24 bits of the dimension-0 lower bound's
// key.  Sorting by class first keeps extents of
// similar size together, so that one long extent does not widen the boxes
// of a leaf of short ones; the order is a heuristic (node bounds come from
// the coordinates whatever the order).  hist[class] counts the extents.
__global__ void __launch_bounds__(kThreads)
k_validate_class(int d, const float* __restrict__ lo, const float* __restrict__ hi, uint32_t cnt,
                 uint32_t* __restrict__ k32, uint32_t* __restrict__ hist, float2* __restrict__ aos,
                 Status* __restrict__ st) {
  __shared__ uint32_t s_h[256];
  for (int i = threadIdx.x; i < 256; i += blockDim.x) s_h[i] = 0u;
  __syncthreads();
  bool bad = false;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    float side = 0.0f;
    for (int k = 0; k < d; ++k) {
      const float a = __ldg(lo + (size_t)k * cnt + i);
      const float b = __ldg(hi + (size_t)k * cnt + i);
      bad |= !(a <= b);
      side = fmaxf(side, b - a);
      if (aos) aos[(size_t)i * d + k] = make_float2(a, b);
    }
    const uint32_t cls = (__float_as_uint(side) >> 23) & 0xffu;
    k32[i] = (cls << kLocalityBits) | (float_key(__ldg(lo + i)) >> kLocalityDrop);
    atomicAdd(&s_h[cls], 1u);
  }
  if (__ballot_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&st->err, kErrExtent);
  __syncthreads();
  for (int i = threadIdx.x; i < 256; i += blockDim.x)
    if (s_h[i]) atomicAdd(&hist[i], s_h[i]);
}

// Instance (batched set, or size class) of every position: the b with
// off[b] <= i < off[b+1] (some b for offsets that are no prefix sums).  A warp fills kFillSpan consecutive positions: one
// search over the offsets (32 places a step), then 32 positions at a time, a
// lane walking on from the last instance found; so one very large instance is
// filled by the whole grid, and the pass is bound by its stores (a binary
// search per position took 188 us for 2.9e7 positions of 4,096 instances).
constexpr uint32_t kFillSpan = 1024;
__global__ void __launch_bounds__(kThreads)
k_fill_inst(const unsigned long long* __restrict__ off, uint32_t count, uint32_t total,
            uint32_t* __restrict__ inst) {
  const uint32_t lane = threadIdx.x & 31u, warps = gridDim.x * (blockDim.x / 32u);
  for (size_t i0 = (size_t)(blockIdx.x * (blockDim.x / 32u) + threadIdx.x / 32u) * kFillSpan;
       i0 < total; i0 += (size_t)warps * kFillSpan) {
    OwnerWalk<const unsigned long long*> owner(off, count, warp_owner(off, count, i0));
    const size_t end = min(i0 + kFillSpan, (size_t)total);
#pragma unroll 4
    for (size_t i = i0 + lane; i < end; i += 32u) inst[i] = owner.at(i);
  }
}

__global__ void __launch_bounds__(kThreads)
k_validate_batch(int d, const float* __restrict__ lo, const float* __restrict__ hi, uint32_t cnt,
                 const uint32_t* __restrict__ inst, unsigned long long* __restrict__ keys,
                 uint32_t* __restrict__ vals, uint32_t* __restrict__ k32, float2* __restrict__ aos,
                 Status* __restrict__ st) {
  bool bad = false;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    for (int k = 0; k < d; ++k) {
      const float a = __ldg(lo + (size_t)k * cnt + i);
      const float b = __ldg(hi + (size_t)k * cnt + i);
      bad |= !(a <= b);
      if (aos) aos[(size_t)i * d + k] = make_float2(a, b);
    }
    const uint32_t key = float_key(__ldg(lo + i)) >> kLocalityDrop;
    if (k32) {
      k32[i] = key;
    } else {
      keys[i] = ((unsigned long long)inst[i] << kLocalityBits) | key;
      vals[i] = i;
    }
  }
  if (__ballot_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&st->err, kErrExtent);
}

__global__ void k_batch_groups(const unsigned long long* __restrict__ off, uint32_t count,
                               const int* __restrict__ glog2, uint32_t* __restrict__ ngroups) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const uint32_t n = (uint32_t)(off[i + 1] - off[i]);
    const int g = glog2[i];
    // g == 0 (no re-sort): the whole instance is one group whose keys are
    // all equal, so the stable sort keeps it in place.  With g >= 6 every
    // instance has at most n / 64 + 1 groups.
    ngroups[i] = g > 0 ? ((n + (1u << g) - 1) >> g) : (n > 0 ? 1u : 0u);
  }
}

__global__ void __launch_bounds__(kThreads)
k_rekey_batch(const uint32_t* __restrict__ vals, const float* __restrict__ lo_k, uint32_t cnt,
              const uint32_t* __restrict__ inst, const unsigned long long* __restrict__ off,
              const int* __restrict__ glog2, const unsigned long long* __restrict__ gbase,
              unsigned long long* __restrict__ keys, int id_bits) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < cnt; i += stride) {
    const uint32_t b = inst[i];
    const int g = glog2[b];
    const uint32_t id = vals[i];
    unsigned long long k;
    if (g == 0) {  // one group, equal keys: the instance keeps its order
      k = gbase[b] << kLocalityBits;
    } else {
      const unsigned long long local = i - off[b];
      const unsigned long long group = gbase[b] + (local >> g);
      k = (group << kLocalityBits) | (float_key(__ldg(lo_k + id)) >> kLocalityDrop);
    }
    keys[i] = id_bits ? (k << id_bits) | id : k;
  }
}

uint32_t grid_for(uint32_t cnt, int sms) {
  uint32_t blocks = (cnt + kThreads - 1) / kThreads;
  const uint32_t cap = (uint32_t)sms * 8u;
  return blocks > cap ? cap : (blocks ? blocks : 1);
}

}  // namespace

cudaError_t launch_rekey(const uint32_t* vals, const float* lo_k, uint32_t cnt, int glog2,
                         unsigned long long* keys, int id_bits, int sms, cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  k_rekey<<<grid_for(cnt, sms), kThreads, 0, s>>>(vals, lo_k, cnt, glog2, keys, id_bits);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_gather(int d, const uint32_t* vals, const float* lo, const float* hi,
                          const float2* aos, uint32_t cnt, float2* qe, uint32_t* qid, int sms,
                          cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  k_gather<<<grid_for(cnt, sms), kThreads, 0, s>>>(d, vals, lo, hi, aos, cnt, qe, qid);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_validate_class(int d, const float* lo, const float* hi, uint32_t cnt,
                                  uint32_t* k32, uint32_t* hist, float2* aos, Status* st, int sms,
                                  cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  k_validate_class<<<grid_for(cnt, sms), kThreads, 0, s>>>(d, lo, hi, cnt, k32, hist, aos, st);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_fill_inst(const unsigned long long* off, uint32_t count, uint32_t total,
                             uint32_t* inst, int sms, cudaStream_t s) {
  if (count == 0 || total == 0) return cudaSuccess;
  const uint32_t warps = (total + kFillSpan - 1) / kFillSpan;
  k_fill_inst<<<grid_for(warps * 32u, sms), kThreads, 0, s>>>(off, count, total, inst);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_validate_batch(int d, const float* lo, const float* hi, uint32_t cnt,
                                  const uint32_t* inst, unsigned long long* keys, uint32_t* vals,
                                  uint32_t* k32, float2* aos, Status* st, int sms, cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  k_validate_batch<<<grid_for(cnt, sms), kThreads, 0, s>>>(d, lo, hi, cnt, inst, keys, vals, k32, aos,
                                                           st);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_batch_groups(const unsigned long long* off, uint32_t count, const int* glog2,
                                uint32_t* ngroups, cudaStream_t s) {
  if (count == 0) return cudaSuccess;
  const uint32_t blocks = (count + 255) / 256 < 1024 ? (count + 255) / 256 : 1024;
  k_batch_groups<<<blocks, 256, 0, s>>>(off, count, glog2, ngroups);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_rekey_batch(const uint32_t* vals, const float* lo_k, uint32_t cnt,
                               const uint32_t* inst, const unsigned long long* off,
                               const int* glog2, const unsigned long long* gbase,
                               unsigned long long* keys, int id_bits, int sms, cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  k_rekey_batch<<<grid_for(cnt, sms), kThreads, 0, s>>>(vals, lo_k, cnt, inst, off, glog2, gbase,
                                                        keys, id_bits);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_validate(int d, const float* lo, const float* hi, uint32_t cnt,
                            uint32_t* k32, bool whole_key, float2* aos, Status* st, int sms,
                            cudaStream_t s) {
  if (cnt == 0) return cudaSuccess;
  if (whole_key)
    k_validate<true><<<grid_for(cnt, sms) + 1u, kThreads, 0, s>>>(d, lo, hi, cnt, k32, aos, st);
  else
    k_validate<false><<<grid_for(cnt, sms), kThreads, 0, s>>>(d, lo, hi, cnt, k32, aos, st);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace ddm
