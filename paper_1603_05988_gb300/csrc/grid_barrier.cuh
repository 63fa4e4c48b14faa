// Bounded grid barrier of the persistent (cooperative) solver kernels.
#pragma once

#include "persist.cuh"
#include "reduce.cuh"

namespace dtr {

constexpr long long kSpinBudget = 4000000000LL;  // ~2 s at 2 GHz
// Largest persistent grid: two buffers of partials per block, 5 x 64 double2 (whole lattice) or 8 x 64 float or double
// (red-black), fit the solver's reduction scratch (kMaxGrid x 5 x 64 double2).
constexpr int kPersistMaxGrid = kMaxGrid / 2;

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Counting grid barrier: arrive, then wait until `target` arrivals in total
// (the barrier's sequence number times the grid size).  Returns false if the
// wait exceeded `budget` clock cycles or another block reported an error.
// Ordering without full fences: thread 0 arrives with a release reduction and
// polls with acquire loads; the block barriers before and after extend that to
// the whole block (the writes of the block's threads happen before the
// release, and the acquire happens before their later reads).
__device__ __forceinline__ bool grid_arrive_wait(GridSync *gs, unsigned int target, long long budget) {
  __shared__ int s_err;
  __syncthreads();
  if (threadIdx.x == 0) {
    s_err = 0;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gs->count) : "memory");
    const long long t0 = clock64();
    while (true) {
      unsigned int c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(&gs->count) : "memory");
      if (c >= target) break;
      if (*(volatile int *)&gs->error) {
        s_err = 1;
        break;
      }
      if (clock64() - t0 > budget) {
        atomicExch(&gs->error, 1);
        s_err = 1;
        break;
      }
    }
  }
  __syncthreads();
  return !s_err;
}

}  // namespace dtr
