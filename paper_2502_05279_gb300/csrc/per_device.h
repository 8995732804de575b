// Things that have to be done once on every device a process uses, such as
// raising a kernel's shared-memory limit: a function-local static would do them
// on the first device only.
#pragma once

#include <atomic>

namespace bmg {

class PerDevice {
  std::atomic<unsigned long long> done_{0};

 public:
  // Calls act() unless it has already succeeded (returned 0) for this device;
  // returns act()'s code, 0 when it was not called.  Threads that get here
  // together may each call it; one that is told 0 without calling it comes after
  // a call that succeeded.
  template <typename F>
  int once(int device, F&& act) {
    const bool kept = device >= 0 && device < 64;
    const unsigned long long bit = kept ? 1ull << device : 0ull;
    if (done_.load(std::memory_order_acquire) & bit) return 0;
    const int rc = act();
    if (rc == 0) done_.fetch_or(bit, std::memory_order_release);
    return rc;
  }
};

}  // namespace bmg
