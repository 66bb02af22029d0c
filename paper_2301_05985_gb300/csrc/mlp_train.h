// mlp_train.h -- launch interface of the learned-start network's training gradient.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

// Loss (mean squared error over rows x 3) and its gradient in the packed parameter order
// W1[216][128], b1[128], W2[128][128], b2, W3[128][128], b3, W4[128][3], b4[3].
struct MlpGradArgs {
  int64_t rows;
  const float* Xf;          // [rows][216] inputs, or null: Xb holds them
  __nv_bfloat16* Xb;        // [rows][224] BF16 inputs (written from Xf when that is given)
  const float* Y;           // [rows][ldy] targets, 3 columns
  int ldy;
  const __nv_bfloat16 *W1, *W2, *W3, *W4;  // [224][128], [128][128] twice, [128][8]
  const float *b1, *b2, *b3, *b4;
  __nv_bfloat16* A[3];      // [rows][128] hidden activations
  __nv_bfloat16* dZ[3];     // [rows][128] gradients at the pre-activations
  __nv_bfloat16* dO;        // [rows][8] gradient at the outputs
  float* part;              // workspace: mlp_grad_part_floats()
  double* loss_part;        // workspace: mlp_grad_max_ctas() doubles
  float* grad;              // [61187]
  double* loss;             // 1
};

// floats of the partials workspace; blocks of the first kernel at most
size_t mlp_grad_part_floats();
int mlp_grad_max_ctas();
cudaError_t launch_mlp_grad(const MlpGradArgs& a, cudaStream_t s);
