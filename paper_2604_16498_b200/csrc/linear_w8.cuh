// The int8-weight linear (linear_w8.cu): entry point for the dispatcher in linear_gelu.cu.
#pragma once

#include <cuda_runtime.h>

namespace forge {

// act((X Wq^T) * scale + b) + residual; arguments as forge_linear_act_w8a16.
int linear_w8(const void* x, const void* w_int8, const float* scale, const void* b, const void* residual, void* y, int M,
              int N, int K, int act, cudaStream_t s);

}  // namespace forge
