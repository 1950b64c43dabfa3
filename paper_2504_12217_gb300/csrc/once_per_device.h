// What every device needs once, such as a kernel's shared-memory limit (an attribute of the
// device that was current when it was set).
#pragma once
#include <atomic>
#include <cstdint>

namespace zkvc {

class OncePerDevice {
 public:
  // f() (a status, 0: done) unless it has succeeded for this device before.  Two threads may
  // run f at once.
  template <class F>
  int operator()(int device, F&& f) {
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
    if (done_.load(std::memory_order_acquire) & bit) return 0;
    const int rc = f();
    if (rc == 0) done_.fetch_or(bit, std::memory_order_release);
    return rc;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace zkvc
