// last_block.cuh -- the block of a grid that finishes last, for reductions that end in the
// launch that makes their partials.
#pragma once

#include <cuda_runtime.h>

// True in every thread of the one block of `total` that arrives last.  Writes to global
// memory that a thread made before the call are visible to that block afterwards (read
// them with __ldcg: another block's lines may sit in this SM's L1).  The counter wraps to
// zero, ready for the next launch; launches that share it must be ordered (one stream).
__device__ __forceinline__ bool last_block(unsigned* ticket, unsigned total) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicInc(ticket, total - 1) == total - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Grid barrier of a cooperative launch: waits until every block has arrived; false in every
// thread of a block whose wait gave up after `polls` polls (< 0: the default, about a second; then *err = 1: device or mapped
// host memory).  `arrived` is zero before the launch; a block that is the last to finish the
// kernel (last_block after the barrier, in every block) sets it back.  Writes made before the
// call by any block are visible after it (read them with __ldcg).
constexpr int kBarrierPolls = 1 << 22;
__device__ __forceinline__ bool grid_barrier(unsigned* arrived, int* err, int polls) {
  __shared__ bool passed;
  if (polls < 0) polls = kBarrierPolls;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    atomicAdd(arrived, 1u);
    bool ok = false;
    for (int i = 0; i < polls && !ok; ++i) {
      unsigned n;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(arrived) : "memory");
      ok = n >= gridDim.x;
    }
    if (!ok) *reinterpret_cast<volatile int*>(err) = 1;
    passed = ok;
  }
  __syncthreads();
  return passed;
}
