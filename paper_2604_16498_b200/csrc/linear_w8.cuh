// The int8-weight linear (linear_w8.cu): plan and entry point for the dispatcher in linear_gelu.cu.
#pragma once

#include <cuda_runtime.h>

namespace forge {

struct W8Plan {
    int nt, tiles_t;   // tokens per tile (a multiple of 16, at most 192), token tiles
    long long tiles;   // of tokens and features
    int split;         // CTAs per tile: 1, 2, 4 or 8
    int own4;          // 4-token pieces that a CTA of a cluster finishes (0 without one)
    int recv_bytes;    // exchange buffer of a CTA
    int groups;        // converter groups: 3 or 4
    int stages;        // of the ring: at least as many as groups
};

// The plan for an M x N output on a GPU with `sms` SMs; false for a size that has none (2^31 tiles or more).
bool linear_w8_plan(int M, int N, int K, int sms, W8Plan* plan);

// act((X Wq^T) * scale + b) + residual; arguments as forge_linear_act_w8a16.
int linear_w8(const void* x, const void* w_int8, const float* scale, const void* b, const void* residual, void* y, int M,
              int N, int K, int act, cudaStream_t s);

}  // namespace forge
