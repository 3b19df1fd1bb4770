// State that the CUDA runtime keeps per device, remembered per device.  No CUDA
// headers: the tests compile it for the host alone.
#pragma once

#include <atomic>
#include <mutex>

namespace rosko {

// The dynamic shared memory limit of a kernel.  cudaFuncSetAttribute acts on
// the current device, and a later call with fewer bytes lowers the limit: each
// device's limit only grows, one thread at a time.
class SmemLimit {
 public:
  // Raise the limit on `dev` (the current device) to `bytes` where it is lower:
  // set(bytes) makes it so and returns whether it could.
  template <class Set>
  bool ensure(int dev, int bytes, Set set) {
    if (dev < 0 || dev >= kDevices) return set(bytes);
    if (have_[dev].load(std::memory_order_acquire) >= bytes) return true;
    std::lock_guard<std::mutex> lk(mu_);
    if (have_[dev].load(std::memory_order_relaxed) >= bytes) return true;
    if (!set(bytes)) return false;
    have_[dev].store(bytes, std::memory_order_release);
    return true;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> have_[kDevices] = {};
  std::mutex mu_;
};

}  // namespace rosko
