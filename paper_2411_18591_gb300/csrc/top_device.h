// What a kernel needs once on each device before it is launched there: its dynamic shared memory allowed,
// and how many of its blocks the device holds at the launch's block shape. Both belong to the device that
// is current, and a process may hold a handle on each of several.
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>
#include <cstddef>

namespace top {

class KernelOnDevices {
 public:
  // Before a launch of `kernel` on the current device; *resident: its blocks there at once (0 if unknown).
  cudaError_t ready(const void* kernel, int threads, size_t smem, int* resident) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev < kDevices;
    int known = kept ? resident1_[dev].load(std::memory_order_acquire) : 0;
    if (known == 0) {
      if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
        if (e != cudaSuccess) return e;
      }
      int sms = 0, per_sm = 0;
      if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
          cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(&per_sm, kernel, threads, smem, cudaOccupancyDefault) !=
              cudaSuccess)
        sms = 0;
      known = sms * per_sm + 1;
      if (kept) resident1_[dev].store(known, std::memory_order_release);
    }
    *resident = known - 1;
    return cudaSuccess;
  }
  template <class K>
  cudaError_t ready(K* kernel, int threads, size_t smem, int* resident) {
    return ready(reinterpret_cast<const void*>(kernel), threads, smem, resident);
  }

 private:
  static constexpr int kDevices = 64;             // beyond them the set-up is done at every launch
  std::atomic<int> resident1_[kDevices] = {};  // blocks at once + 1; 0: not set up yet
};

}  // namespace top
