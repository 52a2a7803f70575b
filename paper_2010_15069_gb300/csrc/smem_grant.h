// Dynamic shared memory that a kernel may use beyond the default 48 KB, raised
// before a launch that needs more.  The limit is one per kernel and device and a
// later call overwrites an earlier one, so it is only ever raised, under a mutex:
// a launch on another thread that needs less (the same kernel for another grid or
// another number of modes) never lowers it between a grant and its launch.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <mutex>

namespace spgpe {

class SmemGrant {
 public:
  static constexpr int kDevices = 64;
  // `set(bytes)` is called with the new limit when this device's is below it; a
  // refusal is returned and not remembered.
  template <class Set> cudaError_t raise(int dev, size_t smem, Set set) {
    if (dev < 0 || dev >= kDevices) return cudaErrorInvalidDevice;
    if (granted_[dev].load(std::memory_order_acquire) >= smem) return cudaSuccess;
    std::lock_guard<std::mutex> lk(mu_);
    if (granted_[dev].load(std::memory_order_relaxed) >= smem) return cudaSuccess;
    const cudaError_t e = set(smem);
    if (e == cudaSuccess) granted_[dev].store(smem, std::memory_order_release);
    return e;
  }
  // For the current device.  A refusal does not stay behind as the runtime's last
  // error, which the next launch would report as its own.
  template <class K> cudaError_t operator()(K kern, size_t smem) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
      e = raise(dev, smem, [&](size_t b) {
        return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
      });
    if (e != cudaSuccess) cudaGetLastError();
    return e;
  }

 private:
  std::mutex mu_;
  std::atomic<size_t> granted_[kDevices] = {};
};

}  // namespace spgpe
