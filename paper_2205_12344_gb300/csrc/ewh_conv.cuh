// Launchers of the tensor-core convolutions (ewh_conv.cu).
#pragma once
#include <cuda_runtime.h>

namespace ewh {
cudaError_t launch_conv3x3(const void* x, const void* w, const float* bias, float* pre, void* out, int act, int N,
                           int H, int W, int Ci, int Co, cudaStream_t st);
cudaError_t launch_conv3x3_wgrad(const void* x, const void* dy, float* dw, int N, int H, int W, int Ci, int Co,
                                 cudaStream_t st);
}  // namespace ewh
