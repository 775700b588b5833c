// tpx_mlp_train.cuh -- the fused training step of the perceptron refiner.
#pragma once

#include <cuda_runtime.h>

namespace tpxt {
constexpr int kMaxHidden = 160;   // widths beyond this take the general GEMMs (tpx_refine.cu)
// one Adam step on n rows; work: n (4 h + 12) floats
cudaError_t train_step(cudaStream_t s, float *P, float *M, float *V, float *G, int h, long long step, const float *x,
                       const float *y, long long n, float lr, float w_off, float *work, float *loss);
}  // namespace tpxt
