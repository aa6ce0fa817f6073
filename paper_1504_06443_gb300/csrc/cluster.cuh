// Bounded waits of the kernels whose CTAs push to each other's shared memory (tri.cu, tridiag_cluster.cu,
// panel_cluster.cu).
#pragma once
#include "gep_internal.cuh"

namespace gep {
namespace {

__device__ __forceinline__ uint32_t cta_shared(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Waits up to two seconds for a phase of a barrier that the pushes of other CTAs complete; on expiry records the
// timeout.  DRAIN false: also gives up once an error is recorded.  DRAIN true: for pushes known to be under way,
// before the CTA retires.
template <bool DRAIN>
__device__ __forceinline__ bool cluster_wait(uint32_t bar, uint32_t parity, int* st) {
  unsigned long long t0 = 0, now;
  for (int it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if ((it & 15) != 15) continue;
    if (!DRAIN && *(volatile int*)(st + 1) != 0) return false;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (t0 == 0) t0 = now;
    if (now - t0 > 2000000000ull) {
      atomicExch(st + 1, GEP_ERR_TIMEOUT);
      return false;
    }
  }
}

}  // namespace
}  // namespace gep
