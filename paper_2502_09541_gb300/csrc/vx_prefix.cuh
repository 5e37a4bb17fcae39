// When a prefix sort is worth it, and its repair.  The pairs are in the order of their keys' bits above
// `shift`; what is left are groups of equal prefix whose low bits descend
// somewhere.  Plain functions of positions, which the kernels call and which run
// on the CPU as well (tests/prefix_check.cc).
#pragma once

#include <cmath>
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

// How many low key bytes (4, 3 or 0) a sort may leave to the repair, from m
// sampled rows of n.  c[0], c[1]: sampled keys that differ from another one but
// agree with it in the upper four / five bytes; such keys have to be rare (at
// most kFixRate of them per key among the n).  c[2]: a key that occurs eight
// times in the sample; c[3]: sampled rows that repeat a key.  Keys must not
// repeat much: two keys of nine rows each that share their prefix make a group too
// large to repair.  The sort checks what it finds, so a sample that misleads costs
// a second sort of the pairs and nothing else.  Partitions of 8.4M uniform keys:
// four passes and the repair 0.37 ms, eight passes 0.62; the call of 67M pairs
// 10.2 -> 9.3 ms.
//
// distinct_rows: no row is in the sample twice, so every repeat is one of the
// input's; keys of r rows each give about (r - 1) m^2 / 2n of them, and the line
// lies at r = 4.5, halfway to nine.  (With the other sample's line 3M pairs whose
// keys occur ten times each were sorted twice, 0.96 ms; in full they take 0.77,
// and keys that occur twice 0.62 with the repair.)  Otherwise rows are drawn with
// repetition, and repeats have to be beyond the rows drawn twice.
constexpr double kFixRate = 0.06;

inline int prefix_bytes(const uint64_t (&c)[4], uint64_t m, uint64_t n, bool distinct_rows) {
  if (c[2]) return 0;
  if (distinct_rows) {
    if ((double)c[3] > 3.5 * (double)m * (double)m / (2.0 * (double)n)) return 0;
  } else {
    // sample rows that repeat one drawn before: m less the distinct rows drawn
    const double twice = (double)m + (double)n * std::expm1(-(double)m / (double)n);
    if ((double)c[3] > 1.5 * twice + 6.0 * std::sqrt(twice) + 16.0) return 0;
  }
  const double per = 2.0 / (double)m * ((double)n / (double)m);  // a pair of sample neighbours, in neighbours per key
  return (double)c[0] * per <= kFixRate ? 4 : (double)c[1] * per <= kFixRate ? 3 : 0;
}

}  // namespace vx
