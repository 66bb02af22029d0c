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
