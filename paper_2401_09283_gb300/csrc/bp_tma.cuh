// TMA tile loads and the shared-memory barriers that announce them (sm_103a).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

namespace bpk {

__device__ __forceinline__ unsigned smem_addr(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(unsigned long long* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
               : "memory");
}
// Make freshly initialised barriers visible to the TMA unit.
__device__ __forceinline__ void mbar_init_fence() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect(unsigned long long* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
               "r"(bytes)
               : "memory");
}

// Wait for the phase of the given parity.  Each try suspends the thread in
// hardware until the phase completes or the hinted time (20 us) is over: with
// the short default time the polling itself took a fifth of the issue slots.
// Bounded: false after MBAR_TRIES tries.  A try lasts 2 to 3 us whatever the hint
// (1024 of "10 ms" were over after 3 ms, which memory that has to be paged in could
// exceed): 2^20 of them are 2 to 3 s, and 20 s at most.  (A limit by the timer in place of the
// count made the forward spill, 256^3 x 248 3.28 against 3.33 ms.)
#ifdef BP_BOUNDS_CHECK
constexpr int MBAR_TRIES = 1 << 14;  // a test lets it run out
#else
constexpr int MBAR_TRIES = 1 << 20;
#endif
__device__ __forceinline__ bool mbar_wait(unsigned long long* bar, unsigned parity) {
  const unsigned a = smem_addr(bar);
  unsigned ok = 0;
#pragma unroll 1
  for (int i = 0; i < MBAR_TRIES; ++i) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(a), "r"(parity), "r"(20000u)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// One box of a 3D tensor map to shared memory; completion counts on bar.
// Elements outside the tensor arrive as zeros.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z,
                                            unsigned long long* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cta.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(dst)),
      "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
      : "memory");
}

}  // namespace bpk
