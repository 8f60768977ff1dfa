// C entry point of the decode step on fp16 tensors.  The kernels are in attn_decode.cuh.
#include "attn_decode.cuh"

extern "C" int forge_attn_decode_splitkv_f16(const void* q, const void* k_cache, const void* v_cache, void* out,
                                             int B, int Hq, int Hkv, int Smax, int D,
                                             const int32_t* lens, int num_splits, float scale,
                                             void* workspace, size_t workspace_bytes, void* stream) {
    return forge::decode_splitkv_impl<true>(q, k_cache, v_cache, out, B, Hq, Hkv, Smax, D, lens, num_splits, scale,
                                            workspace, workspace_bytes, stream);
}
