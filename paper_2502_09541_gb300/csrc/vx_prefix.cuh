// Repair of a prefix sort: the pairs are in the order of their keys' bits above
// `shift`; what is left are groups of equal prefix whose low bits descend
// somewhere.  Plain functions of positions, which the kernels call and which run
// on the CPU as well (tests/prefix_check.cc).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define VX_HD __host__ __device__ __forceinline__
#else
#define VX_HD inline
#endif

namespace vx {

constexpr uint32_t kFixGroup = 16;  // pairs of a group that one thread repairs

// A thread's positions i with a neighbour i + 1 < n, a stride apart: 64 bits, so
// that the last step of an n near 2^32 does not wrap
struct PrefixWalk {
  uint64_t i, n, stride;
  VX_HD bool more() const { return i + 1 < n; }
  VX_HD void next() { i += stride; }
};

enum PrefixFind { kFixNone, kFixList, kFixFull };

// What the neighbours i, i + 1 < n ask for: a group is listed, with its first
// pair, at its first descent; a group with a descent and more than kFixGroup
// pairs asks for the sort in full.
VX_HD PrefixFind prefix_find(const uint64_t *k, uint64_t n, uint64_t i, int shift, uint64_t *first) {
  const uint64_t a = k[i], c = k[i + 1], prefix = a >> shift;
  if (a <= c || c >> shift != prefix) return kFixNone;
  uint32_t size = 2;  // pairs of the group seen
  uint64_t j = i;
  for (uint64_t x = a; j > 0; --j) {  // back to the group's first pair, or to an earlier descent
    const uint64_t y = k[j - 1];
    if (y >> shift != prefix) break;
    if (y > x) return kFixNone;
    if (++size > kFixGroup) return kFixFull;
    x = y;
  }
  for (uint64_t e = i + 2; e < n && k[e] >> shift == prefix; ++e)
    if (++size > kFixGroup) return kFixFull;
  *first = j;
  return kFixList;
}

// a stable insertion sort of the group that starts at `first`, where it is
VX_HD void prefix_fix(uint64_t *k, uint32_t *v, uint64_t n, uint64_t first, int shift) {
  const uint64_t prefix = k[first] >> shift;
  for (uint64_t e = first + 1; e < n && k[e] >> shift == prefix; ++e) {
    const uint64_t x = k[e];
    const uint32_t y = v[e];
    uint64_t at = e;
    for (; at > first && k[at - 1] > x; --at) {
      k[at] = k[at - 1];
      v[at] = v[at - 1];
    }
    k[at] = x;
    v[at] = y;
  }
}

}  // namespace vx
