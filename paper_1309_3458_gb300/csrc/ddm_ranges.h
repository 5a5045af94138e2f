// Index arithmetic of batched sets: which instance owns a position, chunk or
// leaf.  The offsets are the caller's device arrays and not checked (they are
// documented to be prefix sums that end at the set's size), so everything here
// stays inside the arrays whatever they hold.  Plain C++, so that a host
// program can run it over offsets that no GPU should see.
#ifndef DDM_RANGES_H
#define DDM_RANGES_H
#include <stdint.h>

#ifdef __CUDACC__
#define DDM_HD __host__ __device__ __forceinline__
#else
#define DDM_HD inline
#endif

namespace ddm {

// Search for the b with prefix[b] <= i < prefix[b + 1], by a warp: 32 places a
// step.  Every lane probes its place; take() gets the lanes that answered yes.
struct OwnerSearch {
  uint32_t lo, hi;  // prefix[lo] <= i < prefix[hi], for a prefix sum from 0 on
  DDM_HD explicit OwnerSearch(uint32_t count) : lo(0), hi(count) {}
  DDM_HD bool more() const { return hi - lo > 1u; }
  DDM_HD uint32_t step() const { return (hi - lo + 31u) / 32u; }
  template <typename Prefix>
  DDM_HD bool probe(const Prefix& prefix, uint32_t lane, unsigned long long i) const {
    const uint32_t at = lo + lane * step();
    return at < hi && prefix[at] <= i;
  }
  DDM_HD void take(uint32_t yes) {
    const uint32_t s = step();
    uint32_t last = 0;  // highest lane; none (offsets that do not start at 0): lane 0
#ifdef __CUDA_ARCH__
    if (yes) last = 31u - (uint32_t)__clz((int)yes);
#else
    for (uint32_t l = 0; l < 32u; ++l)
      if (yes >> l & 1u) last = l;
#endif
    lo += last * s;
    hi = hi < lo + s ? hi : lo + s;
  }
};

// Owners of ascending positions, from instance b (which owns one no later) on:
// the next few instances one by one, behind a longer run of empty ones a search.
template <typename Prefix>
struct OwnerWalk {
  Prefix prefix;
  uint32_t count, b;
  unsigned long long next;  // first position behind instance b; none behind the last
  DDM_HD OwnerWalk(Prefix p, uint32_t n, uint32_t from) : prefix(p), count(n) { enter(from); }
  DDM_HD void enter(uint32_t to) {
    b = to;
    next = to + 1u < count ? prefix[to + 1u] : ~0ull;
  }
  DDM_HD uint32_t at(unsigned long long i) {
    for (int steps = 0; next <= i; ++steps) {
      if (steps < 8) {
        enter(b + 1u);
        continue;
      }
      uint32_t lo = b, hi = count;  // prefix[lo] <= i < prefix[hi]
      while (hi - lo > 1u) {
        const uint32_t mid = lo + (hi - lo) / 2u;
        if (prefix[mid] <= i) lo = mid; else hi = mid;
      }
      enter(lo);
      break;
    }
    return b;
  }
};

}  // namespace ddm
#endif  // DDM_RANGES_H
