// dot4.cuh -- a step of the FP32 running sums of the inner Krylov solve.
#pragma once

#include <cmath>
#include <cuda_runtime.h>

// s + a . b.  The four products meet first, so a thread's running sum rounds once per float4:
// 43 times over 20.0 M unknowns on 456 blocks of 256 threads.  As a chain of four fused
// multiply-adds into s it rounded 171 times there, and the sum of a long chain is off by the
// roundings at the sum's own size.
__host__ __device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
  return s + fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, a.w * b.w)));
}
