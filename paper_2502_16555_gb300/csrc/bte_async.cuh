// mbarriers with bounded waits and bulk copies between global and shared memory.
#pragma once

#include <cstdint>

#include "bte_kernels.h"

namespace bte {

constexpr long long kWaitCycles = 1ll << 32;   // bounded device waits, about 2 s
constexpr long long kProbeCycles = 1ll << 21;  // about 1 ms: the wait of BTE_FLAG_DIAG_HARMONIC_TIMEOUT

__device__ __forceinline__ uint32_t saddr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(saddr(b)), "r"(count));
}

__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(saddr(b)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded; false if it ran out. On expiry the status bit is set, later waits of the CTA on phases that are
// not complete return at once, and the kernel runs to its end on whatever the buffers hold (every access
// stays in bounds); the step reports it. The thread that issues a barrier's copies or products also waits
// for them: when its own wait fails it issues nothing more, and it waits again (mbar_drain) for what is
// in flight, so that nothing lands in memory that the CTA has given back.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, volatile int* gave_up, unsigned* status,
                                          long long limit = kWaitCycles) {
  if (mbar_try(b, parity)) return true;
  const long long t0 = clock64();
  while (!*gave_up) {
    if (mbar_try(b, parity)) return true;
    if (clock64() - t0 > limit) {
      *gave_up = 1;
      atomicOr(status, kTimeout);
    }
  }
  return false;
}

__device__ __forceinline__ void mbar_drain(uint64_t* b, uint32_t parity) {
  const long long t0 = clock64();
  while (!mbar_try(b, parity) && clock64() - t0 < kWaitCycles) {
  }
}

// global -> shared, completion counted on bar; shared -> global in this thread's bulk group
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(saddr(dst)),
               "l"(src), "r"(bytes), "r"(saddr(bar))
               : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(saddr(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(bar)), "r"(bytes) : "memory");
}

}  // namespace bte
