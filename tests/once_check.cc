// OncePerDevice (csrc/vx_once.h): once for every device, again after a failure.
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>

#include "vx_once.h"

#define CHECK(x)                                          \
  do {                                                    \
    if (!(x)) {                                           \
      std::printf("%s:%d: %s\n", __FILE__, __LINE__, #x); \
      std::exit(1);                                       \
    }                                                     \
  } while (0)

int main() {
  vx::OncePerDevice once;
  int calls[66] = {};
  for (int round = 0; round < 3; ++round)
    for (int d = 0; d < 66; ++d) CHECK(once.run(d, [&] { return ++calls[d] > 1 || d != 5; }) == (d != 5 || round > 0));
  for (int d = 0; d < 64; ++d) CHECK(calls[d] == (d == 5 ? 2 : 1));
  CHECK(calls[64] == 3 && calls[65] == 3);
  vx::OncePerDevice shared;
  std::atomic<int> n{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&] {
      for (int i = 0; i < 1000; ++i) shared.run(i % 4, [&] { return n.fetch_add(1) >= 0; });
    });
  for (auto &t : ts) t.join();
  CHECK(n >= 4 && n <= 32);
  std::printf("ok\n");
  return 0;
}
