// Launchers of the tensor-core convolutions (ewh_conv.cu).
#pragma once
#include <cuda_runtime.h>

namespace ewh {

// The waits of a convolution CTA that gave up, before it returns its shared and
// tensor memory: no load may land there any more, no MMA read or write it.  Steps
// [multiplied, issued) were requested but no MMA waited for them (barrier full of
// their stage); the commit after the last MMAs covers those of earlier steps (empty of
// its stage, `done` after the last of all steps).  A stage's barriers complete one phase
// every `stages` steps.
enum CvBar { CV_FULL, CV_EMPTY, CV_DONE };
template <class Wait>
__host__ __device__ inline void cv_drain(int issued, int multiplied, int steps, int stages, Wait wait) {
  for (int s = multiplied; s < issued; ++s) wait(CV_FULL, s % stages, (unsigned)(s / stages) & 1u);
  const int last = multiplied - 1;
  if (last < 0) return;
  if (multiplied < steps)
    wait(CV_EMPTY, last % stages, (unsigned)(last / stages) & 1u);
  else
    wait(CV_DONE, 0, 0u);
}

cudaError_t launch_conv3x3(const void* x, const void* w, const float* bias, float* pre, void* out, int act, int N,
                           int H, int W, int Ci, int Co, cudaStream_t st);
cudaError_t launch_conv3x3_wgrad(const void* x, const void* dy, float* dw, int N, int H, int W, int Ci, int Co,
                                 cudaStream_t st);
}  // namespace ewh
