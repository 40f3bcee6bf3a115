// Training of the closure network on the CUDA cores (mlp_train.cu): launchers
// used by the C entry points in closure.cu.
#pragma once

#include <cuda_runtime.h>

namespace fftk {

constexpr int kNP = 9094;  // parameters of the 5-64-64-64-6 network

// blocks (and so gradient partials of kNP floats and loss partials) of a
// gradient over at most B samples; never falls as B grows
int mlp_grad_blocks(long long B);

// Adam's constants for one step: c1, c2 the bias corrections
struct AdamStep {
  float* params;
  float* m;
  float* v;
  float lr, b1, b2, eps, c1, c2;
};

cudaError_t launch_mlp_grad(bool bf16, const float* params, const float* x, const float* t, int B, float* part,
                            double* loss_part, cudaStream_t st);
// the gradient from the partials (fixed order, FP64), the loss when asked
// for, and with `adam` the parameter update from that gradient
cudaError_t launch_mlp_reduce(int B, const float* part, const double* loss_part, float* grad, double* loss,
                              const AdamStep* adam, cudaStream_t st);
cudaError_t launch_mlp_forward_cc(bool bf16, const float* params, const float* x, float* y, int B, cudaStream_t st);
cudaError_t launch_adam(const AdamStep& a, const float* grad, cudaStream_t st);

}  // namespace fftk
