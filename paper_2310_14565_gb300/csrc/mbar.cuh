// Shared-memory barriers of the asynchronous copies and their bounded waits
// (the multiply-accumulate kernels).
#pragma once
#include "common.cuh"

__device__ __forceinline__ u64 globaltimer_ns() {
  u64 t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(u32 addr, u32 count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(u32 addr, u32 bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(u32 addr) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(u32 addr, u32 parity) {
  u32 ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(addr), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for phase `parity` of an mbarrier for at most about one second.  The
// clock is read every 256 tries only: a read of %globaltimer is slow enough to
// delay a wait that is about to end.
__device__ __forceinline__ bool mbar_wait_bounded(u32 addr, u32 parity) {
  u64 t0 = 0;
  for (u32 i = 1; !mbar_try_wait(addr, parity); ++i) {
    if (i & 255) continue;
    const u64 now = globaltimer_ns();
    if (!t0) t0 = now;
    if (now - t0 > 1000000000ull) return false;
  }
  return true;
}
