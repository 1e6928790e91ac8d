// 3x3x3 convolutions of the learned warm start (nn_conv.cu): the forward
// pass, its data gradient (sign = -1 with the transposed weights) and its
// weight and bias gradients.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace rt3d {

// Co in {16, 32, 48, 64, 96}, Ci a multiple of 16
cudaError_t launch_conv3d(const __nv_bfloat16 *X, const __nv_bfloat16 *Wt, const float *bias,
                          __nv_bfloat16 *Y, float *Yf, int S, int nx, int ny, int nz, int Ci, int Co,
                          bool relu, int sign, cudaStream_t s);
// Ci, Co multiples of 16; db nullable
cudaError_t launch_conv3d_wgrad(const __nv_bfloat16 *X, const __nv_bfloat16 *dY, float *dW, float *db,
                                int S, int nx, int ny, int nz, int Ci, int Co, cudaStream_t s);

}  // namespace rt3d
