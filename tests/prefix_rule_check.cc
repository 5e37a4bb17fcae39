// Whether a sample of 4,096 rows sends a pair sort to the prefix sort
// (prefix_bytes, csrc/vx_prefix.cuh), for keys that occur r times each.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <random>
#include <vector>

#include "vx_prefix.cuh"

static int choice(uint64_t n, uint64_t r, uint64_t mask, unsigned seed) {
  std::mt19937_64 rng(seed);
  std::vector<uint64_t> keys(n);
  for (uint64_t i = 0; i < n; i += r) {
    const uint64_t k = rng() & mask;
    for (uint64_t j = i; j < std::min(n, i + r); ++j) keys[j] = k;
  }
  std::shuffle(keys.begin(), keys.end(), rng);
  const uint64_t m = std::min<uint64_t>(n, 4096);
  std::map<uint64_t, int> rows;
  uint64_t c[4] = {0, 0, 0, 0};
  for (uint64_t i = 0; i < m; ++i) {
    const int seen = ++rows[keys[i * n / m]];
    c[3] += seen > 1;
    c[2] += seen == 8;
  }
  for (auto a = rows.begin(), b = std::next(a); b != rows.end(); a = b++) {
    c[0] += a->first >> 32 == b->first >> 32;
    c[1] += a->first >> 24 == b->first >> 24;
  }
  return vx::prefix_bytes(c, m, n, true);
}

int main() {
  int bad = 0;
  for (unsigned seed = 1; seed <= 3; ++seed)
    for (uint64_t n : {32768ull, 100003ull, 1000000ull, 3000017ull})
      for (uint64_t r : {1ull, 2ull, 10ull, 20ull, 200ull}) {
        const int want = r <= 2 ? 4 : 0, got = choice(n, r, ~0ull, seed);
        if (got != want) std::printf("n %llu, %llu rows a key: %d\n", (unsigned long long)n, (unsigned long long)r, got), ++bad;
      }
  if (choice(1000000, 1, 0xFFFFFFFFull, 1) != 0) std::printf("32-bit keys\n"), ++bad;
  if (!bad) std::printf("ok\n");
  return bad != 0;
}
