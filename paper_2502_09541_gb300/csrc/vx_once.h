// Work that is needed once per device of a process (tests/once_check.cc).
#pragma once

#include <atomic>
#include <cstdint>

namespace vx {

class OncePerDevice {
 public:
  // Runs f() unless it has succeeded for this device before; whether it has now.
  // Threads that come at the same time may each run it.
  template <class F>
  bool run(int device, F &&f) {
    const uint64_t bit = device >= 0 && device < 64 ? 1ull << device : 0;  // others: every time
    if (done_.load(std::memory_order_acquire) & bit) return true;
    if (!f()) return false;
    done_.fetch_or(bit, std::memory_order_release);
    return true;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace vx
