// Grid-wide barrier of the cooperative kernels (every CTA of the launch is
// resident, which cudaLaunchCooperativeKernel guarantees or refuses).
#pragma once

#include "cb_internal.cuh"

namespace cb {

__device__ __forceinline__ uint64_t grid_now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(uint32_t *p, uint32_t v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// A barrier gives up after wait_ns of global time (kGridWaitNs but in tests) or
// kGridPolls polls; the CTA arrives at no further one, so the others give up at
// their next at the latest.
constexpr uint64_t kGridWaitNs = 4000000000ull;
constexpr uint32_t kGridPolls = 1u << 27;

// One thread's wait for *ctr to reach `target` (a count that only grows).
__device__ __forceinline__ bool grid_wait(const uint32_t *ctr, uint32_t target, uint64_t wait_ns) {
  if (ld_acquire(ctr) >= target) return true;
  const uint64_t t0 = grid_now_ns();
  for (uint32_t it = 1; it < kGridPolls; ++it) {
    if (ld_acquire(ctr) >= target) return true;
    if ((it & 255u) == 0 && grid_now_ns() - t0 > wait_ns) return false;
  }
  return false;
}

// Barrier over `ctas` CTAs, all resident; every thread of each calls it.  *ctr is 0
// before the launch; `epoch` counts the caller's barriers.  Writes made before
// it by any of their threads are visible after it.  Returns false (in every
// thread of the CTA) when the wait gave up.
__device__ __forceinline__ bool grid_sync(uint32_t *ctr, uint32_t &epoch, uint32_t ctas, uint64_t wait_ns) {
  epoch += 1;
  bool ok = true;
  __syncthreads();
  if (ctas > 1 && threadIdx.x == 0) {
    red_release(ctr, 1u);  // with the barrier above: after every store of the CTA
    ok = grid_wait(ctr, epoch * ctas, wait_ns);  // acquire; the barrier below passes it on
  }
  return __syncthreads_and(ok) != 0;
}

}  // namespace cb
