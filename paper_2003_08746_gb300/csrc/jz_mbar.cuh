// Shared-memory mbarriers (inline PTX) with bounded waits, for the fused FP32-flux kernel's TMA copies
// (jz_stage32.cu).
#pragma once

#include <cuda_runtime.h>

namespace jz {

__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_init(unsigned long long* b, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
// Wait for an mbarrier phase with a bounded number of polls; false if it never completed.
constexpr int kWaitPolls = 1 << 18;   // ~1 s on GB300 (each unanswered try_wait suspends a few microseconds)
__device__ __forceinline__ bool wait_bar(unsigned long long* bar, unsigned parity) {
  const unsigned b = smem_u32(bar);
  for (int it = 0; it < kWaitPolls; ++it) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(b), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

}  // namespace jz
