// A grid barrier for cooperative launches, every wait bounded.
#pragma once

#include "bse_internal.cuh"

namespace bse {

constexpr long long GRID_SPIN = 1ll << 22;   // polls of one barrier wait

__device__ __forceinline__ unsigned int ld_acquire_u32(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// All CTAs of the launch meet here; false (in every thread of the CTA) when the wait expired.  The
// arrivals of all barriers of a launch add up in one counter, so nothing is reset and a waiter
// polls the counter itself: one release and the polls, 1.3 us where an arrival count that the last
// CTA turns into a generation number, with a fence in every thread, took 2.2.
__device__ __forceinline__ bool grid_sync(GridBar* gb, unsigned int nblk, unsigned int& gen, int* s_ok) {
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned int target = (gen + 1) * nblk;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&gb->count) : "memory");
    long long i = 0;
    while ((int)(ld_acquire_u32(&gb->count) - target) < 0) {
      if (++i > GRID_SPIN) {
        atomicExch(&gb->err, 1);
        ok = 0;
        break;
      }
    }
    *s_ok = ok;
  }
  ++gen;
  __syncthreads();
  return *s_ok != 0;
}

}  // namespace bse
