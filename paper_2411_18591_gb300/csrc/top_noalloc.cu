// The static device scratch of top_propagate_noalloc, in a translation unit of its own: its
// module (and so the array) is loaded on a device only when this unit's symbol is first used
// there (the first no-alloc call), or for every context when CUDA loads modules eagerly
// (CUDA_MODULE_LOADING=EAGER). Processes that only use handle calls never pay for it under the
// default lazy loading.
#include <mutex>

#include "top_aux.h"

namespace top {

static __device__ __align__(256) unsigned char g_noalloc_scratch[TOP_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int kNoallocDevices = 64;
std::mutex g_mutex;
NoallocScratch g_scratch[kNoallocDevices] = {};
}  // namespace

cudaError_t noalloc_scratch(NoallocScratch* out, bool load) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kNoallocDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_mutex);
  NoallocScratch& s = g_scratch[dev];
  if (!s.mem && load) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    if (!p) return cudaErrorInvalidSymbol;
    // host memory is mapped here once, also when the thread is capturing a stream
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    e = fault_word(&s.fault, &s.fault_dev);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e != cudaSuccess) return e;
    s.mem = p;
  }
  *out = s;
  return cudaSuccess;
}

cudaError_t fault_word(int** host, int** device) {
  void* word = nullptr;
  void* mapped = nullptr;
  cudaError_t e = cudaHostAlloc(&word, sizeof(int), cudaHostAllocMapped);
  if (e != cudaSuccess) return e;
  e = cudaHostGetDevicePointer(&mapped, word, 0);
  if (e != cudaSuccess) {
    cudaFreeHost(word);
    return e;
  }
  *host = static_cast<int*>(word);
  **host = 0;
  *device = static_cast<int*>(mapped);
  return cudaSuccess;
}

}  // namespace top
