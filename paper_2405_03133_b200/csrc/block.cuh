// RMSNorm and residual kernels for the layer inside a pre-norm residual block (Section 4.1: LLaMA blocks).
#pragma once
#include "common.cuh"

namespace lory {

// x_hat = x / sqrt(mean_j x_j^2 + eps) * gamma per token; inv_rms [tokens] is kept for the backward.
template <typename T>
int launch_rmsnorm(const T* x, const T* gamma, T* x_hat, float* inv_rms, long tokens, int d, float eps,
                   cudaStream_t st);
// dx = RMSNorm backward of dxh (gradient wrt x_hat) + dy (the residual path); dgamma = sum over tokens of
// dxh * x * inv_rms (added to the stored value when accumulate != 0).  slab: float [block_norm_slabs(tokens), d].
template <typename T>
int launch_rmsnorm_backward(const T* x, const T* gamma, const float* inv_rms, const T* dxh, const T* dy, T* dx,
                            T* dgamma, float* slab, long tokens, int d, int accumulate, cudaStream_t st);
int block_norm_slabs(long tokens);

}  // namespace lory
