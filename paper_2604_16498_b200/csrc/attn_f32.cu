// Fused attention with fp32 tensors (Eq. 8 / Eq. 9): one kernel computes scores, mask, online softmax and the product with
// V; scores and probabilities stay on chip.  Plain fp32 FMA arithmetic (no tensor cores) so that the result stays within
// 1e-4 of an fp64 evaluation.
//
// What bounds it: for a single short prompt (12 heads x 128 x 128 x 64) the latency of one CTA's chain of copies, dot
// products and reductions; for larger batches the shared-memory reads that feed the FMAs.  So a warp works on a 16 x 32
// tile of scores with 4 rows x 4 keys per thread (8 16-byte reads feed 64 FMAs, issued as 32 packed pairs), and the
// eight warps of a CTA share the keys of a tile: KSPLIT warps take different keys of the same 16 rows, each with its own
// running maximum and sum, and are merged once at the end.
//   KSPLIT = 8: 16 query rows per CTA, 16 keys of a 128-key tile per warp: shortest chain, most CTAs
//   KSPLIT = 2: 64 query rows per CTA, 32 keys of a 64-key tile per warp: K and V are copied a quarter as often
// Thread = rows 4 (lane / 8) .. + 3 of its warp's 16, keys lane % 8 + 8 j; in P V the same rows, head columns
// 4 (lane % 8) .. + 3 and + 32 h.  Q is multiplied by scale * log2(e) on its way to shared memory, so that products which fp32
// holds only after scaling do not overflow before it.
// 12 heads, D = 64, causal, cold inputs, against 16-row CTAs of four warps with one row x 8 keys per thread: 1 x 128
// 12.1 -> 7.0 us, 3 x 200 42.7 -> 18.7 us, 8 x 512 278 -> 122 us; error against fp64 2.1e-7 -> 1.5e-7 (shorter sums).
#include "forge_common.cuh"

namespace forge {
namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kPad = 4;      // floats of padding per Q and K row: eight keys side by side read eight different bank groups
constexpr int kPStride = 20; // floats between the keys of a warp's P tile (16 rows each)

template <int D, int KSPLIT>
struct Tile {
    static constexpr int BN = KSPLIT == 8 ? 128 : 64;   // keys per tile
    static constexpr int KW = BN / KSPLIT;              // keys per warp and tile: 16 or 32
    static constexpr int NJ = KW / 8;                   // keys per thread
    static constexpr int BM = 16 * kWarps / KSPLIT;     // query rows per CTA
    static constexpr int LD = D + kPad;
    static constexpr int kQ = 0;                        // offsets in floats
    static constexpr int kK = kQ + BM * LD;
    static constexpr int kV = kK + BN * LD;
    static constexpr int kP = kV + BN * D;
    static constexpr int kML = kP + kWarps * KW * kPStride;  // per warp and row: maximum, sum
    static constexpr int kBytes = (kML + kWarps * 16 * 2) * 4;
    // the warps' partial outputs are merged where K and V were
    static_assert(kWarps * 16 * D <= BN * LD + BN * D, "merge buffer");
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    const int bytes = valid ? 16 : 0;  // the rest is zero-filled
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// two fp32 FMAs in one instruction
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
    float2 d;
    asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\t"
        "mov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\tmov.b64 rc, {%6, %7};\n\t"
        "fma.rn.f32x2 rd, ra, rb, rc;\n\t"
        "mov.b64 {%0, %1}, rd;\n\t}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}

template <int D, int KSPLIT>
__global__ void __launch_bounds__(kThreads, D == 64 ? 2 : 1)
attn_f32_kernel(const float* __restrict__ q, const float* __restrict__ k, const float* __restrict__ v,
                float* __restrict__ out, int Hq, int Hkv, int Sq, int Skv, int mask_kind,
                const int32_t* __restrict__ lens, float scale_log2) {
    using T = Tile<D, KSPLIT>;
    constexpr int LD = T::LD, NJ = T::NJ, DV = D / 32;
    extern __shared__ __align__(16) float smem_f32[];
    float* sQ = smem_f32 + T::kQ;
    float* sK = smem_f32 + T::kK;
    float* sV = smem_f32 + T::kV;
    float* sML = smem_f32 + T::kML;

    pdl_launch_dependents();  // the next kernel may move in; nothing global is touched before the previous one is done
    pdl_wait();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ks = warp % KSPLIT, group = warp / KSPLIT;  // which keys, which 16 rows
    const int rg = lane >> 3, kg = lane & 7;
    const int q0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * T::BM;  // longest (causal) first
    const int h = blockIdx.y, b = blockIdx.z;
    const int kvh = h / (Hq / Hkv);
    float* sP = smem_f32 + T::kP + warp * T::KW * kPStride;

    int kvlen = Skv;
    if (mask_kind & FORGE_MASK_PADDING) kvlen = min(max(lens[b], 0), Skv);
    const int causal_off = Skv - Sq;
    const bool causal = (mask_kind & FORGE_MASK_CAUSAL) != 0;
    // keys that the CTA / this warp's rows can see at all: the last row sees the most
    int kv_end = kvlen, kv_end_warp = kvlen;
    const int w0 = q0 + group * 16;  // first row of this warp
    if (causal) {
        kv_end = min(kv_end, min(q0 + T::BM, Sq) + causal_off);
        kv_end_warp = min(kv_end_warp, min(w0 + 16, Sq) + causal_off);
    }
    if (w0 >= Sq) kv_end_warp = 0;

    const float* qb = q + ((size_t)(b * Hq + h) * Sq + q0) * D;
    const float* kb = k + (size_t)(b * Hkv + kvh) * Skv * D;
    const float* vb = v + (size_t)(b * Hkv + kvh) * Skv * D;

    // keys at and beyond kv_end are zero-filled, never read (padding may hold anything)
    auto copy_tile = [&](int j0) {
        for (int idx = tid; idx < T::BN * (D / 4); idx += kThreads) {
            const int r = idx / (D / 4), c = idx % (D / 4);
            cp_async16(sK + r * LD + c * 4, kb + (j0 + r < kv_end ? (size_t)(j0 + r) * D + c * 4 : 0), j0 + r < kv_end);
        }
        cp_async_commit();
        for (int idx = tid; idx < T::BN * (D / 4); idx += kThreads) {
            const int r = idx / (D / 4), c = idx % (D / 4);
            cp_async16(sV + r * D + c * 4, vb + (j0 + r < kv_end ? (size_t)(j0 + r) * D + c * 4 : 0), j0 + r < kv_end);
        }
        cp_async_commit();
    };
    constexpr int kQPieces = T::BM * (D / 4) / kThreads;
    float4 qpiece[kQPieces];
#pragma unroll
    for (int i = 0; i < kQPieces; ++i) {
        const int idx = i * kThreads + tid, r = idx / (D / 4), c = idx % (D / 4);
        qpiece[i] = q0 + r < Sq ? *reinterpret_cast<const float4*>(qb + (size_t)r * D + c * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (kv_end > 0) copy_tile(0);
#pragma unroll
    for (int i = 0; i < kQPieces; ++i) {
        const int idx = i * kThreads + tid, r = idx / (D / 4), c = idx % (D / 4);
        *reinterpret_cast<float4*>(sQ + r * LD + c * 4) =
            make_float4(qpiece[i].x * scale_log2, qpiece[i].y * scale_log2, qpiece[i].z * scale_log2, qpiece[i].w * scale_log2);
    }

    float m_run[4], l_run[4];
    float2 acc[4][2 * DV];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        m_run[i] = -INFINITY;
        l_run[i] = 0.f;  // of this thread's keys only, until the end
#pragma unroll
        for (int d = 0; d < 2 * DV; ++d) acc[i][d] = make_float2(0.f, 0.f);
    }

    for (int j0 = 0; j0 < kv_end; j0 += T::BN) {
        if (j0 > 0) {
            __syncthreads();  // the previous tile has been consumed
            copy_tile(j0);
        }
        cp_async_wait<1>();
        __syncthreads();
        const int key0 = j0 + ks * T::KW;
        const bool work = key0 < kv_end_warp;
        if (work) {
            float2 s2[4][NJ];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) s2[i][j] = make_float2(0.f, 0.f);
            const float* qr = sQ + (group * 16 + rg * 4) * LD;
            const float* kr = sK + (ks * T::KW + kg) * LD;
#pragma unroll 4
            for (int c = 0; c < D; c += 4) {
                float4 qv[4], kv[NJ];
#pragma unroll
                for (int i = 0; i < 4; ++i) qv[i] = *reinterpret_cast<const float4*>(qr + i * LD + c);
#pragma unroll
                for (int j = 0; j < NJ; ++j) kv[j] = *reinterpret_cast<const float4*>(kr + j * 8 * LD + c);
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < NJ; ++j) {
                        s2[i][j] = ffma2(make_float2(qv[i].x, qv[i].y), make_float2(kv[j].x, kv[j].y), s2[i][j]);
                        s2[i][j] = ffma2(make_float2(qv[i].z, qv[i].w), make_float2(kv[j].z, kv[j].w), s2[i][j]);
                    }
            }
            float p[NJ][4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int limit = min(kvlen - 1, causal ? w0 + rg * 4 + i + causal_off : 0x7fffffff);  // last visible key
                float s[NJ], m_tile = -INFINITY;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    s[j] = key0 + kg + 8 * j <= limit ? s2[i][j].x + s2[i][j].y : -INFINITY;
                    m_tile = fmaxf(m_tile, s[j]);
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) m_tile = fmaxf(m_tile, __shfl_xor_sync(0xffffffffu, m_tile, o));
                const float m_new = fmaxf(m_run[i], m_tile);
                // a row that has seen no key yet keeps m = -inf; use 0 as the reference to avoid inf - inf
                const float m_ref = m_new == -INFINITY ? 0.f : m_new;
                const float alpha = exp2f(m_run[i] - m_ref);  // 0 when m_run = -inf
                m_run[i] = m_new;
                l_run[i] *= alpha;
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    p[j][i] = exp2f(s[j] - m_ref);  // masked: exp2(-inf) = 0 exactly
                    l_run[i] += p[j][i];
                }
#pragma unroll
                for (int d = 0; d < 2 * DV; ++d) { acc[i][d].x *= alpha; acc[i][d].y *= alpha; }
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j)
                *reinterpret_cast<float4*>(sP + (kg + 8 * j) * kPStride + rg * 4) = make_float4(p[j][0], p[j][1], p[j][2], p[j][3]);
        }
        cp_async_wait<0>();
        __syncthreads();  // V has landed (and P is complete)
        if (work) {
            const float* vr = sV + ks * T::KW * D + kg * 4;
            // A hidden key has a probability of exactly 0, but 0 x NaN is NaN: a warp stops at the last key that any of its 16 rows
            // sees.  (With 16 rows per CTA the copy stops there already.)
            const int nk = T::BM > 16 ? min(T::KW, kv_end_warp - key0) : T::KW;
#pragma unroll 4
            for (int j = 0; j < nk; ++j) {
                const float4 pv = *reinterpret_cast<const float4*>(sP + j * kPStride + rg * 4);
                const float pr[4] = {pv.x, pv.y, pv.z, pv.w};
#pragma unroll
                for (int d = 0; d < DV; ++d) {
                    const float4 vv = *reinterpret_cast<const float4*>(vr + j * D + d * 32);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i][2 * d] = ffma2(make_float2(pr[i], pr[i]), make_float2(vv.x, vv.y), acc[i][2 * d]);
                        acc[i][2 * d + 1] = ffma2(make_float2(pr[i], pr[i]), make_float2(vv.z, vv.w), acc[i][2 * d + 1]);
                    }
                }
            }
        }
    }

    // Merge the KSPLIT warps of every 16 rows.
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) l_run[i] += __shfl_xor_sync(0xffffffffu, l_run[i], o);
        if (kg == 0) *reinterpret_cast<float2*>(sML + (warp * 16 + rg * 4 + i) * 2) = make_float2(m_run[i], l_run[i]);
    }
    __syncthreads();  // every warp is done with K and V
    float* merge = sK;  // [warp][16 rows][D]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int r = rg * 4 + i;
        float m_all = -INFINITY, l_all = 0.f;
#pragma unroll
        for (int w = 0; w < KSPLIT; ++w) m_all = fmaxf(m_all, sML[((group * KSPLIT + w) * 16 + r) * 2]);
        const float m_ref = m_all == -INFINITY ? 0.f : m_all;
#pragma unroll
        for (int w = 0; w < KSPLIT; ++w) {
            const float2 ml = *reinterpret_cast<const float2*>(sML + ((group * KSPLIT + w) * 16 + r) * 2);
            l_all += ml.y * exp2f(ml.x - m_ref);
        }
        // this warp's share of the row, normalised (no visible key: zeros)
        const float f = l_all > 0.f ? exp2f(m_run[i] - m_ref) / l_all : 0.f;
#pragma unroll
        for (int d = 0; d < DV; ++d)
            *reinterpret_cast<float4*>(merge + (warp * 16 + r) * D + kg * 4 + d * 32) =
                make_float4(acc[i][2 * d].x * f, acc[i][2 * d].y * f, acc[i][2 * d + 1].x * f, acc[i][2 * d + 1].y * f);
    }
    __syncthreads();
    float* ob = out + ((size_t)(b * Hq + h) * Sq + q0) * D;
    for (int idx = tid; idx < T::BM * (D / 4); idx += kThreads) {
        const int r = idx / (D / 4), c = idx % (D / 4);
        if (q0 + r >= Sq) break;
        float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int w = 0; w < KSPLIT; ++w) {
            const float4 x = *reinterpret_cast<const float4*>(merge + (((r >> 4) * KSPLIT + w) * 16 + (r & 15)) * D + c * 4);
            o.x += x.x; o.y += x.y; o.z += x.z; o.w += x.w;
        }
        *reinterpret_cast<float4*>(ob + (size_t)r * D + c * 4) = o;
    }
}

template <int D, int KSPLIT>
int launch_f32(const float* q, const float* k, const float* v, float* out, int B, int Hq, int Hkv, int Sq, int Skv,
               int mask_kind, const int32_t* lens, float scale_log2, cudaStream_t s) {
    using T = Tile<D, KSPLIT>;
    const dim3 grid((Sq + T::BM - 1) / T::BM, Hq, B);
    // A grid of no more CTAs than SMs takes shared memory for one per SM: launched early, beside the previous kernel's CTAs, two of them would
    // share an SM that is free already while others fall idle a moment later.  1 x 12 x 128 without and with it, us: back to back 7.7 and
    // 5.5, between two linears 6.4 and 5.5, on two streams 8.2 and 7.1 a pair; 1 x 12 x 64 5.1 and 4.9, on two streams 6.1 and 5.1.
    constexpr int kAlone = 116 * 1024;
    const int smem = T::kBytes < kAlone && (long long)grid.x * Hq * B <= sm_count() ? kAlone : T::kBytes;
    FORGE_SET_SMEM_ONCE((attn_f32_kernel<D, KSPLIT>), T::kBytes < kAlone ? kAlone : T::kBytes);
    FORGE_CUDA_TRY(launch_pdl(attn_f32_kernel<D, KSPLIT>, grid, dim3(kThreads), smem, s, q, k, v, out, Hq, Hkv, Sq, Skv,
                              mask_kind, lens, scale_log2));
    return finish_launch(1);
}

}  // namespace
}  // namespace forge

extern "C" int forge_attn_fused_f32(const void* q, const void* k, const void* v, void* out,
                                    int B, int Hq, int Hkv, int Sq, int Skv, int D,
                                    int mask_kind, const int32_t* lens, float scale, void* stream) {
    using namespace forge;
    int st = check_attn_args(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens);
    if (st != FORGE_OK) return st;
    if (Hq > 65535 || B > 65535) return FORGE_ERR_UNSUPPORTED;
    const float scale_log2 = scale * 1.4426950408889634f;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const float* qf = static_cast<const float*>(q);
    const float* kf = static_cast<const float*>(k);
    const float* vf = static_cast<const float*>(v);
    float* of = static_cast<float*>(out);
    // Tall tiles once 16-row ones would come to more than about 5.5 per SM: with 768 of them the two are level or the short
    // ones ahead (8 x 128: 19.7 / 19.1 us; 2 x 512 padded: 42.0 / 48.1), with 912 the tall ones are (4 x 300, D = 128:
    // 73.5 / 63.9; 8 x 512: 142 / 122).
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    const bool wide = (long long)((Sq + 15) / 16) * Hq * B > 11LL * sms / 2;
    if (D == 64)
        return wide ? launch_f32<64, 2>(qf, kf, vf, of, B, Hq, Hkv, Sq, Skv, mask_kind, lens, scale_log2, s)
                    : launch_f32<64, 8>(qf, kf, vf, of, B, Hq, Hkv, Sq, Skv, mask_kind, lens, scale_log2, s);
    return wide ? launch_f32<128, 2>(qf, kf, vf, of, B, Hq, Hkv, Sq, Skv, mask_kind, lens, scale_log2, s)
                : launch_f32<128, 8>(qf, kf, vf, of, B, Hq, Hkv, Sq, Skv, mask_kind, lens, scale_log2, s);
}
