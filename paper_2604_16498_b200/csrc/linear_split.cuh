// The fused linear with K split over clusters (linear_split.cu): entry points for the dispatcher in linear_gelu.cu.
#pragma once

#include <cuda_runtime.h>

namespace forge {

struct SplitPlan {
    int bn;           // accumulator columns of a tile: 64 or 128
    int split;        // CTAs per tile: 1, 2, 4 or 8
    bool two_per_sm;  // ring of about 100 KB instead of 220 KB
};

// The plan for one row tile (M <= 128).
SplitPlan linear_split_plan_row(bool gated, int M, int N, int K, int sms);

// Several row tiles: true (and the plan) when this kernel is expected to beat the pair kernel (linear_pair.cu).
bool linear_split_plan_rows(int M, int N, int K, int sms, SplitPlan* plan);

// act(x W + b) + residual; arguments as forge_linear_act (f16: fp16 instead of bf16 tensors).
int linear_split(const SplitPlan& plan, bool f16, const void* x, const void* w, const void* b, const void* residual, void* y,
                 int M, int N, int K, int act, int w_layout, cudaStream_t s);

// silu(x Wg) * (x Wu) (bf16); arguments as forge_linear_swiglu.
int linear_split_swiglu(const SplitPlan& plan, const void* x, const void* w_gate, const void* w_up, void* y, int M, int N,
                        int K, int w_layout, cudaStream_t s);

}  // namespace forge
