// Dynamic shared memory past 48 KB has to be allowed for a kernel before it is
// launched with it, on each device.
#pragma once

#include <atomic>
#include <cstdint>
#include <cuda_runtime_api.h>

namespace p4q {

// One per kernel, beside its launch. allow() sets the kernel's limit on the
// current device, the first time that it is called there; bytes is the largest
// that any launch asks for, so that threads that set it together set the same.
class SmemLimit {
 public:
  template <class Kernel>
  cudaError_t allow(Kernel* kernel, size_t bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0;  // further devices: set on every call
    if (done_.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel), cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(bytes));
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_relaxed);
    return e;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace p4q
