// mlp_tc.h -- tensor-core (tcgen05) inference of the learned-start network.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

// Operand image of the network: the BF16 weights as the MMAs read them from shared memory
// (K-major 8 x 8 core matrices of 128 contiguous bytes: element (k, n) of a layer of width K
// at mlp_core_off(n, k, K / 8 * 128)) and the FP32 biases; one bulk copy brings it in.
constexpr int kMlpK1 = 224, kMlpHid = 128, kMlpN4 = 16;  // input and output widths, padded
constexpr uint32_t kMlpCore = 128;
constexpr uint32_t kMlpImgW1 = 0;                                       // [128 n][224 k]
constexpr uint32_t kMlpImgW2 = kMlpImgW1 + kMlpHid * kMlpK1 * 2;        // [128][128]
constexpr uint32_t kMlpImgW3 = kMlpImgW2 + kMlpHid * kMlpHid * 2;
constexpr uint32_t kMlpImgW4 = kMlpImgW3 + kMlpHid * kMlpHid * 2;       // [16][128]
constexpr uint32_t kMlpImgB = kMlpImgW4 + kMlpN4 * kMlpHid * 2;         // b1, b2, b3 [128], b4 [16]
constexpr uint32_t kMlpImgBytes = kMlpImgB + 4 * (3 * kMlpHid + kMlpN4);
static_assert(kMlpImgBytes % 16 == 0, "bulk copy size");

__host__ __device__ inline uint32_t mlp_core_off(int r, int k, uint32_t sbo) {
  return (uint32_t)(r >> 3) * sbo + (uint32_t)(k >> 3) * kMlpCore + (uint32_t)(r & 7) * 16u + (uint32_t)(k & 7) * 2u;
}

struct MlpTcArgs {
  int64_t rows;
  const float* Xf;          // [rows][216] standardised features, FP32 (rounded to BF16 here), or null:
  const __nv_bfloat16* X;   // [rows][224] BF16 (columns >= 216 zero), 16-byte aligned
  const uint8_t* img;       // operand image, 16-byte aligned
  float* out;               // [rows][ldo]: columns 0..2 written
  int ldo;
  int* err;                 // = 1 when a wait gave up (device or mapped host memory)
};

// out = the network's output for every row (GELU hidden layers, BF16 operands and
// activations, FP32 accumulation)
cudaError_t launch_mlp_infer_tc(const MlpTcArgs& a, cudaStream_t s);
