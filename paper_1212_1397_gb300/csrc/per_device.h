// Settings that a kernel keeps per device (its dynamic shared memory limit), made once on each device that
// the process uses.  No CUDA in here, so that it runs on the host as well.
#pragma once

#include <stdint.h>

#include <atomic>

namespace helm6 {

class OncePerDevice {
 public:
  // True once set() has returned true for this device, now or in an earlier call; a failure is not kept.
  // Threads that come here together may each call set(), which has to allow that.
  template <class Set>
  bool operator()(int device, Set set) {
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;  // beyond: set each time
    if (done_.load(std::memory_order_acquire) & bit) return true;
    if (!set()) return false;
    done_.fetch_or(bit, std::memory_order_release);
    return true;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace helm6
