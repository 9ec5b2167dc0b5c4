// Asynchronous copies into shared memory for the step kernels (sm_100-class
// PTX): bulk tensor copies (TMA) completing on an mbarrier, and the mbarrier
// operations with a bounded wait.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace hyb {

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

// makes initialised barriers visible to the async (TMA) proxy
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// orders this thread's earlier accesses (and those ordered before them) before
// later async-proxy accesses: to the block's shared memory, or to global
// memory (which costs about a microsecond, so once per item and not per plane)
__device__ __forceinline__ void fence_proxy_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() { asm volatile("fence.proxy.async.global;" ::: "memory"); }

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}

// Arrive on the barrier (release: this thread's earlier accesses, and those
// ordered before them by a warp barrier, happen before the phase completes).
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Limit of the waits that drain a block's own copies before it exits.
constexpr long long kDrainCycles = 1LL << 29;

// Wait for the phase with the given parity of the barrier to complete, for
// at most `budget` clock cycles, giving up early once *abort is nonzero
// (another block timed out).  Returns false on timeout or abort.  A negative
// budget only tests the phase once.  No suspend-time hint on the tries: with
// one the threads sleep past their planes' arrival (257^3 refined, eight
// sources: 468 / 516 us a forward / transposed level against 462 / 509).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long budget, const int* abort) {
  const uint32_t a = smem_addr(bar);
  if (budget < 0) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    return done != 0;
  }
  const long long t0 = clock64();
  for (unsigned it = 1;; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((it & 7) == 0 && (clock64() - t0 > budget || *(const volatile int*)abort != 0)) return false;
  }
}

// ---- the sweep kernel's waits and copies ----
// Limit of its waits that do not depend on other blocks: a block's own copies
// and its own warps.
constexpr long long kOwnCycles = 1LL << 31;

// One try (the hardware may suspend the thread for a short while): has the
// phase with the given parity of the barrier completed?
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// A wait for at most `budget` clock cycles, giving up early once *abort is
// nonzero (a wait timed out; nullptr: not looked at), after a try that failed; a
// negative budget gives up at once.  Out of line, so that the waits in the row
// loops stay short.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, long long budget, const int* abort) {
  if (budget < 0) return false;
  const long long t0 = clock64();
  for (unsigned it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 15) == 0 && (clock64() - t0 > budget || (abort && *(const volatile int*)abort != 0))) return false;
  }
}

// The same for the service warps, which leave the issue slots to the row warps
// between tries.
static __device__ __noinline__ bool mbar_wait_idle(uint64_t* bar, uint32_t parity, long long budget, const int* abort) {
  if (mbar_try(bar, parity)) return true;
  if (budget < 0) return false;
  const long long t0 = clock64();
  for (unsigned it = 1;; ++it) {
    __nanosleep(40);
    if (mbar_try(bar, parity)) return true;
    if ((it & 15) == 0 && (clock64() - t0 > budget || (abort && *(const volatile int*)abort != 0))) return false;
  }
}

// Bulk copy of `bytes` (a multiple of 16) from global to shared memory, both
// 16-byte aligned, completing on the barrier.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// Tiled 3-D bulk tensor copy of one box into shared memory, completing
// (bytes) on the barrier.  x must be a multiple of 16 bytes / element size.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(smem_addr(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}

// Programmatic dependent launch: let the next launch in the stream start its
// blocks now (they wait in pdl_wait), and wait for the previous launch's
// completion and memory before touching what it wrote or read.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

}  // namespace hyb
