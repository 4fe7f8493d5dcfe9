// grid.cuh -- the barrier of the cooperative kernels.
#pragma once

#include "common.cuh"

namespace emst {

constexpr int kBarrierSpins = 1 << 22;
constexpr int kAcquirePolls = 8;

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
      // An acquiring load empties the SM's L1, so a CTA that waits long polls
      // without: it made every step of a chain walk of another CTA an L2 access
      // (30,000 points on a line through emst_compute 10,060 -> 4,170 us).  The
      // first polls, which see the end of most waits, acquire: a fence after
      // them instead cost 0.4 us a barrier (333 points 121 -> 132 us).
      while (v < target) {
        if (spins < kAcquirePolls)
          asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        else
          asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
        if (++spins > kBarrierSpins) {
          atomicOr(status, kErrSpin);
          ok = 0;
          break;
        }
      }
      if (spins > kAcquirePolls)
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// A cooperative launch of at most `grid` CTAs: launch(g) launches g of them.
// Refused as too large (the GPU holds fewer at once than the caller counted,
// as where the SMs are shared out under it) it is made again with half the
// CTAs, down to one; the kernels work with any number.
template <class Launch>
cudaError_t launch_cooperative(int64_t grid, Launch &&launch) {
  for (;;) {
    const cudaError_t e = launch((unsigned)grid);
    if (e != cudaErrorCooperativeLaunchTooLarge || grid <= 1) return e;
    cudaGetLastError();
    grid = (grid + 1) / 2;
  }
}

}  // namespace emst
