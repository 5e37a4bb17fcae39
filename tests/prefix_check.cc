// The repair of a prefix sort (csrc/vx_prefix.cuh) on the CPU: every position of
// a prefix-ordered array asked in turn, as the kernels' threads do.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <numeric>
#include <random>
#include <vector>

#include "vx_prefix.cuh"

using namespace vx;

#define CHECK(x)                                          \
  do {                                                    \
    if (!(x)) {                                           \
      std::printf("%s:%d: %s\n", __FILE__, __LINE__, #x); \
      std::exit(1);                                       \
    }                                                     \
  } while (0)

// groups of equal prefix of the given sizes; kind 0: random low bits, 1: ascending,
// 2: ascending but for the last pair, 3: equal, 4: few values
static void groups(const std::vector<int> &sizes, const std::vector<int> &kinds, int shift, unsigned seed) {
  std::mt19937_64 rng(seed);
  const uint64_t low = (1ull << shift) - 1;
  std::vector<uint64_t> k;
  uint64_t prefix = rng() >> shift >> 20;
  for (size_t g = 0; g < sizes.size(); ++g, prefix += 1 + rng() % 3) {
    std::vector<uint64_t> l(sizes[g]);
    for (auto &x : l) x = kinds[g] == 3 ? 7 : kinds[g] == 4 ? rng() % 3 : 1 + rng() % (low - 1);
    if (kinds[g] == 1 || kinds[g] == 2) std::sort(l.begin(), l.end());
    if (kinds[g] == 2 && l.size() > 1) l.back() = 0;
    for (uint64_t x : l) k.push_back(prefix << shift | x);
  }
  const uint64_t n = k.size();
  std::vector<uint32_t> v(n);
  std::iota(v.begin(), v.end(), 0u);
  std::vector<uint64_t> list;
  uint64_t full = 0;
  for (uint64_t t = 0; t < 7; ++t)
    for (PrefixWalk w{t, n, 7}; w.more(); w.next()) {
      uint64_t first = ~0ull;
      const PrefixFind what = prefix_find(k.data(), n, w.i, shift, &first);
      if (what == kFixList) list.push_back(first);
      full += what == kFixFull;
    }
  std::sort(list.begin(), list.end());
  std::vector<uint64_t> want;
  bool want_full = false;
  uint64_t at = 0;
  for (int size : sizes) {
    if (!std::is_sorted(k.begin() + at, k.begin() + at + size)) {
      if (size <= (int)kFixGroup) want.push_back(at);
      else want_full = true;
    }
    at += size;
  }
  CHECK(list == want);
  CHECK((full != 0) == want_full);
  if (want_full) return;
  std::vector<uint32_t> order(n);
  std::iota(order.begin(), order.end(), 0u);
  std::stable_sort(order.begin(), order.end(), [&](uint32_t a, uint32_t b) { return k[a] < k[b]; });
  std::vector<uint64_t> sorted(n);
  for (uint64_t i = 0; i < n; ++i) sorted[i] = k[order[i]];
  for (uint64_t first : list) prefix_fix(k.data(), v.data(), n, first, shift);
  CHECK(k == sorted);
  CHECK(v == order);
}

int main() {
  for (int shift : {24, 32}) {
    for (int size = 1; size <= 20; ++size)
      for (int kind = 0; kind < 5; ++kind) groups({size}, {kind}, shift, size), groups({3, size, 2}, {0, kind, 2}, shift, size);
    for (unsigned seed = 0; seed < 200; ++seed) {
      std::mt19937 rng(seed);
      std::vector<int> sizes(50), kinds(50);
      for (auto &x : sizes) x = 1 + rng() % (seed % 4 ? 16 : 18);
      for (auto &x : kinds) x = rng() % 5;
      groups(sizes, kinds, shift, seed);
    }
  }
  // the walk ends, in bounds, for pair counts next to 2^32 and the largest grids
  for (uint64_t n : {(1ull << 32) - 1, (1ull << 32) - 311296, (1ull << 32) - 311297, 1ull << 31, 5ull, 2ull, 1ull})
    for (uint64_t stride : {311296ull, 262144ull, 1ull << 20})
      for (uint64_t t : std::vector<uint64_t>{0, 1, 255, stride / 2, stride - 1}) {
        uint64_t steps = 0, last = 0;
        for (PrefixWalk w{t, n, stride}; w.more(); w.next()) {
          CHECK(++steps <= n / stride + 1);
          CHECK(w.i >= last && w.i + 1 < n);
          last = w.i;
        }
        CHECK(steps == (t + 1 < n ? (n - 2 - t) / stride + 1 : 0));
      }
  std::printf("ok\n");
  return 0;
}
