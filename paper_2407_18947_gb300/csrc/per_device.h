// Things that have to be done once for every device of a process, whichever
// thread comes first (a second thread may do them again, without harm).
#pragma once

#include <atomic>

namespace rtcc3 {

class PerDevice {
 public:
  // Runs f() unless it has already returned for this device; device ordinals
  // beyond the mask run it every time, and so does one whose f() threw.
  template <typename F>
  void once(int device, F&& f) {
    const unsigned long long bit = device >= 0 && device < 64 ? 1ULL << device : 0ULL;
    if (bit & done_.load(std::memory_order_acquire)) return;
    f();
    done_.fetch_or(bit, std::memory_order_release);
  }

 private:
  std::atomic<unsigned long long> done_{0};
};

}  // namespace rtcc3
