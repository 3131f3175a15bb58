// A stand-in for the CUDA runtime under the library's objects: "device" memory is host memory, kernels are
// recorded and not run, and a process may have several devices. For tests of what the host side asks of
// the runtime (no GPU needed, and nothing reaches one).
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <cxxabi.h>
#include <vector_types.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "top_internal.h"

namespace {

constexpr int kDevices = 2;

struct Launch {
  std::string name;
  dim3 grid, block;
  size_t smem;
  int device;
  bool refused;
};

int g_device = 0;
bool g_run_out = false;
std::map<const void*, std::string> g_names;                // host function -> kernel
std::map<std::pair<const void*, int>, size_t> g_allowed;   // (host function, device) -> dynamic shared memory
std::vector<Launch> g_launches;
std::map<const void*, void*> g_symbols;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
std::vector<Config> g_configs;
cudaError_t g_last = cudaSuccess;

CUresult encode_tiled(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                      const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                      CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

bool copies_tiles(const std::string& name) {
  return name.find("k_rows_") != std::string::npos && name.find(", true>(") != std::string::npos;
}

}  // namespace

extern "C" {

// ---- what the tests ask
void fake_reset() { g_launches.clear(); }
// From now on every wait of a kernel that moves tiles by copy runs out.
void fake_waits_run_out(int on) { g_run_out = on != 0; }
int fake_launches() { return int(g_launches.size()); }
const char* fake_kernel(int i) { return g_launches[i].name.c_str(); }
int fake_device_of(int i) { return g_launches[i].device; }
int fake_refused(int i) { return g_launches[i].refused; }
void fake_grid(int i, unsigned* xyz) {
  xyz[0] = g_launches[i].grid.x;
  xyz[1] = g_launches[i].grid.y;
  xyz[2] = g_launches[i].grid.z;
}

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  int status = 0;
  char* plain = abi::__cxa_demangle(name, nullptr, nullptr, &status);
  g_names[host] = status == 0 ? plain : name;
  std::free(plain);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  g_configs.push_back({grid, block, smem, static_cast<cudaStream_t>(stream)});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  const Config c = g_configs.back();
  g_configs.pop_back();
  *grid = c.grid;
  *block = c.block;
  *smem = c.smem;
  *static_cast<cudaStream_t*>(stream) = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* kernel, const void* host) {
  *kernel = reinterpret_cast<cudaKernel_t>(const_cast<void*>(host));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t kernel, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t) {
  const void* host = reinterpret_cast<const void*>(kernel);
  Launch l{g_names[host], grid, block, smem, g_device, false};
  const auto allowed = g_allowed.find({host, g_device});
  l.refused = smem > 48 * 1024 && (allowed == g_allowed.end() || allowed->second < smem);
  if (l.refused) {
    g_last = cudaErrorInvalidValue;
  } else if (g_run_out && copies_tiles(l.name)) {
    const auto* p = static_cast<const top::PassParams*>(args[0]);
    if (p->fault) *p->fault = 1;
  }
  g_launches.push_back(l);
  return l.refused ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* host, cudaFuncAttribute, int value) {
  g_allowed[{host, g_device}] = size_t(value);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int threads, size_t, unsigned) {
  *n = threads > 256 ? 1 : 512 / threads;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake runtime error"; }

// ---- devices, memory, streams, events
cudaError_t cudaGetDeviceCount(int* n) { return *n = kDevices, cudaSuccess; }
cudaError_t cudaGetDevice(int* dev) { return *dev = g_device, cudaSuccess; }
cudaError_t cudaSetDevice(int dev) { return g_device = dev, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode*) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = std::aligned_alloc(256, (n + 255) / 256 * 256)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = std::calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { return *d = h, cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  void*& a = g_symbols[symbol];
  if (!a) a = std::aligned_alloc(256, 256);  // kernels that would write it are not run
  return *p = a, cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* found) {
  *fn = reinterpret_cast<void*>(&encode_tiled);
  *found = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = nullptr, cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }

}  // extern "C"
