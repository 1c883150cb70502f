// Opt-in to more dynamic shared memory than the default 48 KB of a block (static memory counts with it).
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdint>

namespace mwk {

// The limit is an attribute of a kernel on one device, and contexts of several devices and threads share a
// process: one SmemLimit per kernel (a function-local static at its launcher) remembers the devices on which it
// has been raised.  `bytes` is the most that any launch of the kernel asks for, always the same value, so threads
// that raise it at the same time set the same limit.  A failure is not remembered; it shows at the launch.
class SmemLimit {
 public:
  template <typename K>
  void raise(K* kernel, size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return;
    const uint64_t bit = dev < 64 ? 1ull << dev : 0;   // further devices set it at every launch
    if (done_.load(std::memory_order_acquire) & bit) return;
    if (cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)bytes) == cudaSuccess)
      done_.fetch_or(bit, std::memory_order_release);
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace mwk
