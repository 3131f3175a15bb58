// Kernel launch, dynamic shared memory and asynchronous-copy spellings used by every unit.
#pragma once

#ifndef TOP_LAUNCH
#define TOP_LAUNCH(kernel, grid, block, smem, stream, ...) kernel<<<(grid), (block), (smem), (stream)>>>(__VA_ARGS__)
#endif

#ifndef TOP_DYN_SMEM
#define TOP_DYN_SMEM(T, name) extern __shared__ __align__(128) T name[]
#endif

#ifndef TOP_ASYNC_COPY
#define TOP_ASYNC_COPY
// 8-byte global -> shared copy that completes asynchronously; both addresses must be 8-byte aligned.
// top_cp_async_wait_all() waits for all of this thread's copies; a block barrier afterwards makes them
// visible to the other threads.
__device__ __forceinline__ void top_cp_async8(void* smem_dst, const void* gsrc) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem_dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gsrc) : "memory");
}
__device__ __forceinline__ void top_cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
#endif

#ifndef TOP_L2_PREFETCH
#define TOP_L2_PREFETCH
// Bring `bytes` (a multiple of 16) from a 16-byte aligned global address into L2, asynchronously.
__device__ __forceinline__ void top_prefetch_l2(const void* gsrc, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(gsrc), "r"(bytes) : "memory");
}
#endif

#ifndef TOP_NAMED_BARRIER
#define TOP_NAMED_BARRIER
// Barrier `id` (1..15) among `count` threads (a multiple of 32, whole warps) of the block.
__device__ __forceinline__ void top_named_barrier(int id, int count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
#endif

#ifndef TOP_TMA
#define TOP_TMA
// Tensor-map copies of 3-D boxes between global and shared memory, completed on an mbarrier (loads) or
// in bulk groups of the issuing thread (stores). Shared addresses are 128-byte aligned, and the
// innermost coordinate times the element size is a multiple of 16 bytes.
__device__ __forceinline__ unsigned top_smem_addr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void top_mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(top_smem_addr(bar)), "r"(count) : "memory");
}
// Makes initialised barriers visible to the copy engine.
__device__ __forceinline__ void top_mbar_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void top_mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared.b64 _, [%0];" ::"r"(top_smem_addr(bar)) : "memory");
}
// Waits for the phase of the given parity to complete, at most `cycles` clock cycles.
__device__ __forceinline__ bool top_mbar_wait(unsigned long long* bar, unsigned parity, long long cycles);
__device__ __forceinline__ void top_mbar_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(top_smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool top_mbar_try(unsigned long long* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;}"
      : "=r"(ok)
      : "r"(top_smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool top_mbar_wait(unsigned long long* bar, unsigned parity, long long cycles) {
  const long long t0 = clock64();
  bool ok = top_mbar_try(bar, parity);
  while (!ok && clock64() - t0 < cycles) ok = top_mbar_try(bar, parity);
  return ok;
}
// Ask the launch for the index of a block that has not started yet (16 bytes of shared memory, 16-byte
// aligned, completed on the mbarrier like a copy); top_ticket reads the answer: the block's x index,
// which this block then runs in its place, or -1 if none is left (ask no more).
__device__ __forceinline__ void top_ask_ticket(void* answer, unsigned long long* bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(
                   top_smem_addr(answer)),
               "r"(top_smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ int top_ticket(const void* answer) {
  unsigned got, x;
  asm volatile(
      "{.reg .pred p;\n\t"
      ".reg .b128 h;\n\t"
      "ld.shared.b128 h, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t"
      "mov.b32 %1, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, h;}"
      : "=r"(got), "=r"(x)
      : "r"(top_smem_addr(answer))
      : "memory");
  return got ? int(x) : -1;
}
__device__ __forceinline__ void top_tma_load3(void* dst, const void* map, int x, int y, int z, unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          top_smem_addr(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(top_smem_addr(bar))
      : "memory");
}
// The same box brought to L2 only.
__device__ __forceinline__ void top_tma_prefetch3(const void* map, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global [%0, {%1, %2, %3}];" ::"l"(map), "r"(x), "r"(y), "r"(z) : "memory");
}
__device__ __forceinline__ void top_tma_store3(const void* map, int x, int y, int z, const void* src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map), "r"(x),
               "r"(y), "r"(z), "r"(top_smem_addr(src))
               : "memory");
}
__device__ __forceinline__ void top_bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// This thread's committed stores: have been read from shared memory / are complete.
__device__ __forceinline__ void top_bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void top_bulk_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Orders this thread's shared-memory writes before later copies that read them.
__device__ __forceinline__ void top_async_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
#endif
