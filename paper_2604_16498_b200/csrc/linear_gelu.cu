// The C entry points of the fused Linear + bias + activation (+ residual) (Listing 6 / Eq. 11) and its variants: argument
// checks and the choice of kernel.  The fp32 accumulator lives in tensor memory; bias and activation are applied to it as
// it is read back, before the single rounding to 16 bits -- the linear output never reaches memory.
//   linear_pair.cu  : 256 x 256 tiles on CTA pairs, for outputs with enough tiles to fill the GPU
//   linear_split.cu : 128 x 64 / 128 x 128 tiles with K split over clusters, for outputs with few tiles
//   linear_w8.cu    : int8 weights with fp16 activations
#include "forge_common.cuh"
#include "linear_pair.cuh"
#include "linear_split.cuh"
#include "linear_w8.cuh"

namespace forge {
namespace {

constexpr int kRowTile = 128;

template <bool F16>
int linear_act_impl(const void* x, const void* w, const void* b, const void* residual, void* y,
                    int M, int N, int K, int act, int w_layout, void* stream) {
    if (!x || !w || !y) return FORGE_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || K <= 0) return FORGE_ERR_INVALID_ARG;
    if (act < FORGE_ACT_GELU_TANH || act > FORGE_ACT_NONE) return FORGE_ERR_INVALID_ARG;
    if (w_layout != FORGE_W_KN && w_layout != FORGE_W_NK) return FORGE_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(w) || !aligned16(y) || (b && !aligned16(b)) || (residual && !aligned16(residual)))
        return FORGE_ERR_INVALID_ARG;
    if ((K % 8) != 0 || (N % 8) != 0) return FORGE_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    // few tiles: K split over clusters (linear_split.cu); large outputs: CTA pairs (linear_pair.cu)
    SplitPlan plan;
    bool split = true;
    if (M <= kRowTile) plan = linear_split_plan_row(false, M, N, K, sms);
    else split = linear_split_plan_rows(M, N, K, sms, &plan);
    return split ? linear_split(plan, F16, x, w, b, residual, y, M, N, K, act, w_layout, s)
                 : linear_pair(F16, x, w, b, residual, y, M, N, K, act, w_layout, s);
}

}  // namespace
}  // namespace forge

extern "C" int forge_linear_act(const void* x, const void* w, const void* b, const void* residual, void* y,
                                int M, int N, int K, int act, int w_layout, void* stream) {
    return forge::linear_act_impl<false>(x, w, b, residual, y, M, N, K, act, w_layout, stream);
}

extern "C" int forge_linear_act_f16(const void* x, const void* w, const void* b, const void* residual, void* y,
                                    int M, int N, int K, int act, int w_layout, void* stream) {
    return forge::linear_act_impl<true>(x, w, b, residual, y, M, N, K, act, w_layout, stream);
}

extern "C" int forge_linear_bias_gelu(const void* x, const void* w, const void* b, void* y,
                                      int M, int N, int K, void* stream) {
    if (!b) return FORGE_ERR_INVALID_ARG;
    return forge_linear_act(x, w, b, nullptr, y, M, N, K, FORGE_ACT_GELU_TANH, FORGE_W_KN, stream);
}

extern "C" int forge_linear_swiglu(const void* x, const void* w_gate, const void* w_up, void* y,
                                   int M, int N, int K, int w_layout, void* stream) {
    using namespace forge;
    if (!x || !w_gate || !w_up || !y) return FORGE_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || K <= 0) return FORGE_ERR_INVALID_ARG;
    if (w_layout != FORGE_W_KN && w_layout != FORGE_W_NK) return FORGE_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(w_gate) || !aligned16(w_up) || !aligned16(y)) return FORGE_ERR_INVALID_ARG;
    if ((K % 8) != 0 || (N % 8) != 0) return FORGE_ERR_UNSUPPORTED;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    // more than one row tile: CTA pairs (linear_pair.cu); else the weight-streaming kernel (linear_split.cu)
    if (M > kRowTile && sms >= 2) return linear_pair_swiglu(x, w_gate, w_up, y, M, N, K, w_layout, s);
    return linear_split_swiglu(linear_split_plan_row(true, M, N, K, sms), x, w_gate, w_up, y, M, N, K, w_layout, s);
}

extern "C" int forge_linear_act_w8a16(const void* x, const void* w_int8, const float* scale, const void* b,
                                      const void* residual, void* y, int M, int N, int K, int act, void* stream) {
    using namespace forge;
    if (!x || !w_int8 || !scale || !y) return FORGE_ERR_INVALID_ARG;
    if (M <= 0 || N <= 0 || K <= 0) return FORGE_ERR_INVALID_ARG;
    if (act < FORGE_ACT_GELU_TANH || act > FORGE_ACT_NONE) return FORGE_ERR_INVALID_ARG;
    if (!aligned16(x) || !aligned16(w_int8) || !aligned16(y) || (b && !aligned16(b)) || (residual && !aligned16(residual)) ||
        (reinterpret_cast<uintptr_t>(scale) & 3u))
        return FORGE_ERR_INVALID_ARG;
    if ((K % 16) != 0 || (N % 8) != 0) return FORGE_ERR_UNSUPPORTED;  // 16-byte rows of int8 weights and of fp16 outputs
    return linear_w8(x, w_int8, scale, b, residual, y, M, N, K, act, static_cast<cudaStream_t>(stream));
}
