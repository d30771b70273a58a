// Barrier of all CTAs of a launch, for kernels that run every step of a call.
//
// A counter in global memory that every CTA adds to once per barrier; every
// wait on it is bounded (about two seconds): on expiry the status word is set,
// an abort word makes every CTA stop at its next barrier, and the launch
// returns (the field is then undefined).  All CTAs are co-resident: such
// kernels go through cooperative launches, which refuse a grid that could not be.
#pragma once
#include <cuda_runtime.h>

#include "internal.h"

namespace bfv {

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Barrier of all CTAs; false when it gave up (timeout, or another CTA's).
// bar[0]: arrivals (want = how many complete this barrier); bar[1]: abort.
// One cluster: the hardware's barrier, which no CTA can miss.
template <bool CLUSTER>
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned want, int *status) {
  if constexpr (CLUSTER) {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
    return true;
  }
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    // release: this CTA's writes (ordered before it by __syncthreads)
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    const long long t0 = clock64();
    while ((int)(ld_acquire_u32(bar) - want) < 0) {  // (the count may wrap)
      if (clock64() - t0 > (1ll << 32)) {
        atomicExch(status, kStatusTimeout);
        atomicExch(bar + 1, 1u);
        ok = 0;
        break;
      }
    }
    if (ld_acquire_u32(bar + 1) != 0) ok = 0;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

}  // namespace bfv
