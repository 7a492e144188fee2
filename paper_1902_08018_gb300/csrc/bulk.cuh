// bulk.cuh -- shared-memory barriers and 1-D bulk copies (global -> shared)
// for the kernels that stage their operands with the copy engine: the
// tensor-core passes (B tiles) and the streamed R = 1 pass (compressed blocks).
#pragma once
#include <cstdint>

namespace whff {
namespace dev {

constexpr uint32_t kMmaSpinLimit = 1u << 22;  // try_wait polls: bounded to seconds

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait; false if the limit ran out.  The in-loop waits of the
// tensor-core kernels take the launch's limit (a handle setting, lowered only
// to test failure detection); the waits before TMEM is freed take the full one.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit = kMmaSpinLimit) {
  for (uint32_t it = 0; it < limit; ++it)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// Bounded wait that also gives up when the CTA's abort flag is raised:
// 1 done, 0 timed out, -1 aborted elsewhere.
__device__ __forceinline__ int mbar_wait_or_abort(uint32_t bar, uint32_t parity, uint32_t limit,
                                                  const volatile int* abort_flag) {
  for (uint32_t it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return 1;
    if (*abort_flag) return -1;
  }
  return 0;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

// One thread: expect `bytes` on `bar` and start the bulk copy global -> shared.
__device__ __forceinline__ void bulk_copy_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

// One thread: expect `bytes` more on `bar` (the copies that bring them follow).
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

// 1-D bulk copy whose bytes the caller has already announced on bar.
__device__ __forceinline__ void bulk_g2s_tx(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}

// 2-D tiled TMA load of the box at (x, y) (x: first column, a multiple of 16
// bytes; y: row) into shared memory (128-byte aligned, 1024 with the 128-byte
// swizzle); completes bytes on bar.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Before a thread's first use of a tensor map in global memory: the map was written
// by a copy, and the unit that reads maps keeps them by address, also from an earlier
// owner of the memory.
__device__ __forceinline__ void tensormap_acquire(const void* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;\n" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}

// Expect `bytes` more on `bar` without arriving.
__device__ __forceinline__ void mbar_expect_tx_only(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}

}  // namespace dev
}  // namespace whff
