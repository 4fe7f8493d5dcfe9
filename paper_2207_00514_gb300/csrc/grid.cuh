// grid.cuh -- the barrier of the cooperative kernels.
#pragma once

#include "common.cuh"

namespace emst {

constexpr int kBarrierSpins = 1 << 22;

// Every CTA adds one to *bar and waits for all of this phase's additions
// (*bar starts at zero; `phase` counts the barriers passed).  The launch is
// cooperative, so all CTAs are resident; the wait is bounded all the same.
// False: gave up (the status says so), and the caller returns.  Everything
// written before the barrier by any CTA is visible after it to plain loads
// (not to loads through the read-only path).
__device__ __forceinline__ bool grid_barrier(uint32_t *bar, uint32_t *status, uint32_t &phase) {
  __shared__ int s_ok;
  __syncthreads();
  ++phase;
  if (threadIdx.x == 0) {
    int ok = 1;
    if (gridDim.x > 1) {
      const uint32_t target = phase * gridDim.x;
      uint32_t v;
      asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(v) : "l"(bar) : "memory");
      v += 1u;
      int spins = 0;
      while (v < target) {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if (++spins > kBarrierSpins) {
          atomicOr(status, kErrSpin);
          ok = 0;
          break;
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

}  // namespace emst
