// mbarriers and bulk copies (inline PTX) shared by the contraction kernels.
// Every wait is bounded: a pipeline wait by a number of tests, a teardown wait
// by the global timer.
#pragma once
#include <stdint.h>

namespace pat {

// Teardown drains (copies and MMAs still in flight after an abort) wait at
// most this long in total, measured on the global timer.
constexpr uint64_t kDrainNs = 2000000000ull;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded pipeline wait for the phase with the given parity: at most `limit`
// tests (mbarrier.try_wait itself suspends the thread for a bounded time, so
// the loop polls without sleeping); false on timeout. limit = 0 gives up at
// once (the plan's wait limit set to 0 exercises the abort path).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i)
    if (mbar_test(bar, parity)) return true;
  return false;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Teardown wait: until the phase completes or the global timer passes
// `deadline` (shared by all drain waits of a thread, so once it has passed the
// remaining drains return at once).
__device__ __forceinline__ bool drain_wait(uint64_t* bar, uint32_t parity, uint64_t deadline) {
  while (!mbar_test(bar, parity))
    if (global_ns() > deadline) return false;
  return true;
}
// Orders this thread's (and, after a barrier, its peers') ordinary shared-memory
// accesses before the asynchronous copies and MMAs it issues next.
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

}  // namespace pat
