// lbm_train.h -- host entry points of the closure-network training kernels
// (lbm_train.cu), called by the C-ABI layer.
#pragma once

#include <cuda_runtime.h>

namespace lbm {

struct MlpShape {
  int H, F, O;   // hidden width, padded feature and output counts
  int valid;     // outputs that enter the loss (3M)
};

// Device scratch of the gradient: the partial gradients [blocks][weights] and
// losses [blocks] of up to `blocks` blocks (one per SM).
struct MlpScratch {
  float* part;
  double* loss;
  int blocks;
};

// Gradient of the mean-squared loss at weights w over `rows` samples
// (features X [rows][F], targets T [rows][O]) into g (packed like w); the loss
// into *d_loss (device).
cudaError_t mlp_train_grad(cudaStream_t s, const MlpShape& sh, const float* w, const float* X, const float* T,
                           int rows, const MlpScratch& z, float* g, double* d_loss);
// One Adam step (step number t >= 1, beta1 0.9, beta2 0.999, eps 1e-8).
cudaError_t mlp_adam(cudaStream_t s, float* w, const float* g, float* m, float* v, long long count, float lr, int t);

}  // namespace lbm
