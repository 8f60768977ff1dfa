// Fused Linear + bias + activation (+ residual) and SwiGLU (Listing 6 / Eq. 11) for outputs with too few tiles to
// fill the GPU: the sum over K of one 128 x BN tile is split over the CTAs of a cluster.
// What bounds it: a single prompt or a batch of decoding sequences streams W once, so the time is that of the bytes of
// W in flight plus a fixed 4-5 us of launch, first copy and last store; a CTA that walks all of K alone keeps one ring
// of tiles in flight while the other SMs idle (16 x 4096 x 14336: 64 CTAs of 224 k-blocks took 38.7 us, 256 CTAs of 56
// take 21.9 us, 5.4 TB/s; 128 x 768 x 3072: 4 CTAs of 48 took 18.6 us, 96 CTAs of 6 take 6.9 us; weights cold).
//
//   grid = tiles x S, a cluster = the S CTAs of one tile; CTA r sums the k-blocks [r, r + 1) * kblocks / S.
//   Each CTA owns BN / S of the tile's output columns.  After its k-loop it sends the other columns of its fp32
//   accumulator to their owners' shared memory (st.shared::cluster), meets the cluster at a barrier, adds the S - 1
//   partial sums it was sent to its own in a fixed order (rank order: results do not depend on timing), applies
//   bias, activation and residual and stores.  S = 1: no cluster, no exchange.  Exchanging through shared memory
//   needs no workspace and no second launch.
//
// Roles: warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-9 epilogue (two per TMEM lane quarter).
// The X tile holds only the rows that exist, rounded up to 8 (xrows): with M = 16 a stage is 2 KB of X and all the
// rest of the ring holds weights, and the copy unit does not fill rows that nobody needs (M = 1 took 23 us where M = 64
// took 14 us with a 128-row box).  The MMA always reads 128 rows of A; those beyond xrows are whatever follows in
// shared memory (inside the allocation) and only reach accumulator rows that nobody reads.
// Where this grid finds room beside the previous kernel's (two CTAs per SM, or CTAs on at most half the SMs), the weights' first
// tiles are asked into L2 before the wait for that kernel, whose tail they overlap (a prefetch into L2 is coherent: it may
// run ahead of a kernel that writes the same lines).  With a CTA of its own on every SM there is no overlap to gain and
// the extra requests cost 0.3-0.6 us.
// A cluster's CTAs wait for one another, so two clusters must not each hold tensor memory that the other one's CTAs wait for.
// Two of these CTAs fit an SM and take at most 256 of its 512 columns; beside a CTA of linear_pair.cu or linear_w8.cu (55000
// registers and more) there is no room for their 23000-31000.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "activations.cuh"
#include "forge_common.cuh"
#include "linear_split.cuh"
#include "sm100_ptx.cuh"
#include "tmap.cuh"

namespace forge {
namespace {

using namespace ptx;

constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + kEpiWarps * 32;
constexpr int kMaxStages = 10;          // deeper rings only lengthen the queue in front of the last tile (13.8 against 14.7 us at 4 x 8192 x 2048 gated)
constexpr int kAhead = 4;                // 8-element pieces of the residual that a thread has in flight
constexpr int kABytes = kBM * kBK * 2;   // what an MMA reads of A

struct SplitParams {
    const uint16_t* bias;
    const uint16_t* residual;  // may be y
    uint16_t* y;
    int M, N, K;
    int act;
    int bn_log2;      // accumulator columns of a tile (gated: gate columns, then up columns)
    int split_log2;   // CTAs per tile
    int xrows;        // rows of the X tile
    int stages;
    int recv_rows;    // rows exchanged (32 .. 128)
    int recv_off, bar_off;  // byte offsets in shared memory
    int prefetch;     // ask for the first weights before the previous kernel is done
    int* status;
};

template <bool F16>
__device__ __forceinline__ uint32_t pack16(float lo, float hi) {
    if constexpr (F16) {
        __half2 v = __floats2half2_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&v);
    } else {
        __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
        return *reinterpret_cast<uint32_t*>(&v);
    }
}
template <bool F16>
__device__ __forceinline__ float widen16(uint16_t bits) {
    if constexpr (F16) return __half2float(__ushort_as_half(bits));
    else return __uint_as_float(static_cast<uint32_t>(bits) << 16);
}

// GATED: tmap_w = gate weights, tmap_w2 = up weights; no bias, residual or activation other than SiLU on the gate.
template <bool W_NK, bool F16, bool GATED>
__global__ void __launch_bounds__(kThreads, 2)
linear_split_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w,
                    const __grid_constant__ CUtensorMap tmap_w2, const SplitParams p) {
    extern __shared__ uint8_t smem_raw[];
    // the same offset in every CTA of the cluster (dynamic shared memory starts at the same address in each)
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.bar_off);
    uint64_t* empty = full + kMaxStages;
    uint64_t* tmem_full = empty + kMaxStages;
    uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(tmem_full + 1);
    float* s_bias = reinterpret_cast<float*>(tmem_full + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int BN = 1 << p.bn_log2;
    const int bno_log2 = GATED ? p.bn_log2 - 1 : p.bn_log2;  // output columns of a tile
    const int S = 1 << p.split_log2;
    const int rank = (int)blockIdx.x & (S - 1);
    const int tile = (int)blockIdx.x >> p.split_log2;
    const int tiles_n = (p.N + (1 << bno_log2) - 1) >> bno_log2;
    const int tile_m = tile / tiles_n;
    const int m0 = tile_m * kBM, n0 = (tile - tile_m * tiles_n) << bno_log2;
    const int kblocks = (p.K + kBK - 1) / kBK;
    const int kb0 = (int)((long long)kblocks * rank >> p.split_log2);
    const int nkb = (int)((long long)kblocks * (rank + 1) >> p.split_log2) - kb0;
    const int a_bytes = p.xrows * (kBK * 2);
    const int stage_bytes = a_bytes + BN * (kBK * 2);

    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        mbar_init(tmem_full, 1);
        fence_mbar_init();
        prefetch_tmap(&tmap_w);
        if constexpr (GATED) prefetch_tmap(&tmap_w2);
        prefetch_tmap(&tmap_x);
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_slot, BN);
        tmem_relinquish();
    }
    // W's tiles of this CTA's kb-th k-block into shared memory at dst / into L2 only
    auto load_w = [&](int kb, uint8_t* dst, uint64_t* bar) {
        const int k0 = (kb0 + kb) * kBK;
        if constexpr (W_NK) {                 // rows of W, 64 K-elements (one swizzle span) each
            tma_load_2d(dst, &tmap_w, bar, k0, n0);
            if constexpr (GATED) tma_load_2d(dst + (BN / 2) * 128, &tmap_w2, bar, k0, n0);
        } else {                              // boxes of 64 K-rows x 64 columns
            for (int c = 0; c < (1 << bno_log2); c += 64) {
                tma_load_2d(dst + c * 128, &tmap_w, bar, n0 + c, k0);
                if constexpr (GATED) tma_load_2d(dst + (BN / 2 + c) * 128, &tmap_w2, bar, n0 + c, k0);
            }
        }
    };
    auto prefetch_w = [&](int kb) {
        const int k0 = (kb0 + kb) * kBK;
        if constexpr (W_NK) {
            tma_prefetch_l2_2d(&tmap_w, k0, n0);
            if constexpr (GATED) tma_prefetch_l2_2d(&tmap_w2, k0, n0);
        } else {
            for (int c = 0; c < (1 << bno_log2); c += 64) {
                tma_prefetch_l2_2d(&tmap_w, n0 + c, k0);
                if constexpr (GATED) tma_prefetch_l2_2d(&tmap_w2, n0 + c, k0);
            }
        }
    };
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_base_slot;
    bool failed = false;
    if (S > 1) cluster_arrive();  // this CTA runs: its shared memory may be written (awaited before the exchange)
    pdl_launch_dependents();
    if (p.prefetch && warp == 0 && elect_one())
        for (int kb = 0; kb < nkb && kb < p.stages; ++kb) prefetch_w(kb);
    pdl_wait();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(&empty[stage], phase ^ 1)) { failed = true; break; }
                uint8_t* sa = smem + stage * stage_bytes;
                mbar_expect_tx(&full[stage], stage_bytes);
                load_w(kb, sa + a_bytes, &full[stage]);
                tma_load_2d(sa, &tmap_x, &full[stage], (kb0 + kb) * kBK, m0);
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idesc = F16 ? make_idesc_f16(kBM, BN, /*a_mn_major=*/false, /*b_mn_major=*/!W_NK)
                                       : make_idesc_bf16(kBM, BN, /*a_mn_major=*/false, /*b_mn_major=*/!W_NK);
            int stage = 0;
            uint32_t phase = 0;
            for (int kb = 0; kb < nkb; ++kb) {
                if (!mbar_wait(&full[stage], phase)) { failed = true; break; }
                const uint32_t sa = smem_u32(smem + stage * stage_bytes);
                const uint32_t sb = sa + a_bytes;
                tc_fence_after_sync();
#pragma unroll
                for (int k = 0; k < kBK / 16; ++k) {
                    // K-major operands: 16 K-elements = 32 bytes further along the 128-byte swizzled row;
                    // MN-major W: 16 K-rows = two 1024-byte groups, 64-column chunks kBK * 128 bytes apart
                    const uint64_t a_desc = make_smem_desc(sa + k * 32, 16, 1024);
                    const uint64_t b_desc = W_NK ? make_smem_desc(sb + k * 32, 16, 1024)
                                                 : make_smem_desc(sb + k * 2048, kBK * 128, 1024);
                    mma_ss(tmem_base, a_desc, b_desc, idesc, (kb | k) != 0);
                }
                mma_commit(&empty[stage]);
                if (++stage == p.stages) { stage = 0; phase ^= 1; }
            }
            if (!failed) mma_commit(tmem_full);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3;             // TMEM lane quarter this warp may access
        const int half = (warp - 2) >> 2;         // takes every other 32-column chunk / 8-column group
        const int etid = (warp - 2) * 32 + lane;
        const int row = quarter * 32 + lane;
        const bool live = quarter * 32 < p.M - m0;  // this warp has rows of the output
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const int own_log2 = bno_log2 - p.split_log2;  // output columns this CTA finishes
        const int own = 1 << own_log2;
        const int own0 = n0 + (rank << own_log2);
        // this warp's 8-column groups of the slice: the first or the second half (a single group: the first warp's)
        const int first = own > 8 ? half * (own >> 4) : 0;
        const int ngroups = own > 8 ? own >> 4 : 1 - half;
        const int segs = GATED ? 2 : 1;
        uint8_t* recv = smem + p.recv_off;
        // bias and residual are fetched while the k-loop runs
        for (int i = etid; i < own; i += kEpiWarps * 32) {
            s_bias[i] = (p.bias != nullptr && own0 + i < p.N) ? widen16<F16>(p.bias[own0 + i]) : 0.f;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kEpiWarps * 32) : "memory");
        const bool row_ok = m0 + row < p.M;
        auto load_residual = [&](int i) {  // 8 elements of group i of this thread's row
            const int col = own0 + (first + i) * 8;
            if (GATED || p.residual == nullptr || i >= ngroups || !row_ok || col >= p.N) return make_uint4(0, 0, 0, 0);
            return *reinterpret_cast<const uint4*>(p.residual + (size_t)(m0 + row) * p.N + col);
        };
        uint4 res[kAhead];
#pragma unroll
        for (int i = 0; i < kAhead; ++i) res[i] = load_residual(i);
        if (!warp_wait(tmem_full, 0)) failed = true;
        tc_fence_after_sync();
        if (S > 1) {
            cluster_wait();  // every CTA of the cluster runs
            if (live && !failed) {
                // recv of the owner: [source slot][segment][4-column chunk][row] of 16 bytes (consecutive rows, i.e. lanes,
                // lie side by side: no bank conflicts on either end)
                const uint32_t recv0 = smem_u32(recv);
                const int chunks_log2 = own_log2 - 2;
#pragma unroll 1
                for (int ch = half; ch < BN / 32; ch += 2) {
                    uint32_t r[32];
                    tmem_ld_x32(taddr + ch * 32, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int c = ch * 32 + j * 4;
                        const int seg = GATED ? c >> bno_log2 : 0;
                        const int oc = c & ((1 << bno_log2) - 1);
                        const int owner = oc >> own_log2;
                        if (owner == rank) continue;
                        const int slot = rank - (rank > owner ? 1 : 0);
                        const int chunk = ((slot * segs + seg) << chunks_log2) + ((oc & (own - 1)) >> 2);
                        const uint32_t dst = map_addr_to_cta(recv0 + (uint32_t)(chunk * p.recv_rows + row) * 16, owner);
                        st_cluster_v4(dst, r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
                    }
                }
            }
            cluster_arrive();
            cluster_wait();  // the other CTAs' partial sums have arrived
        }
        if (live && !failed) {
            // The ring is free (every copy into it has been consumed): each warp collects its 32 rows there, so that rows
            // leave in runs of up to 128 bytes instead of one 16-byte piece per row and store.
            const int pieces_log2 = own > 8 ? own_log2 - 4 : 0;  // 16-byte pieces per row of this warp
            const int pieces = 1 << pieces_log2;
            uint8_t* stage_out = smem + (warp - 2) * (32 * 16) * pieces;
            auto place = [&](int r, int c) { return stage_out + (((r << pieces_log2) + (c ^ ((r >> (3 - pieces_log2)) & (pieces - 1)))) << 4); };
#pragma unroll 1
            for (int i0 = 0; i0 < ngroups; i0 += kAhead) {
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const int i = i0 + u;
                    if (i >= ngroups) break;
                    const int g = first + i;
                    const uint4 r16 = res[u];
                    res[u] = load_residual(i + kAhead);
                    float z[2][8];
#pragma unroll
                    for (int seg = 0; seg < (GATED ? 2 : 1); ++seg) {
                        uint32_t mine[8];
                        tmem_ld_x8(taddr + (seg << bno_log2) + (rank << own_log2) + g * 8, mine);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 8; ++k) z[seg][k] = 0.f;
                        for (int src = 0; src < S; ++src) {  // in rank order
                            if (src == rank) {
#pragma unroll
                                for (int k = 0; k < 8; ++k) z[seg][k] += __uint_as_float(mine[k]);
                            } else {
                                const int slot = src - (src > rank ? 1 : 0);
                                const int chunk = ((slot * segs + seg) << (own_log2 - 2)) + g * 2;
                                const float4 a = *reinterpret_cast<const float4*>(recv + (size_t)(chunk * p.recv_rows + row) * 16);
                                const float4 b = *reinterpret_cast<const float4*>(recv + (size_t)((chunk + 1) * p.recv_rows + row) * 16);
                                z[seg][0] += a.x; z[seg][1] += a.y; z[seg][2] += a.z; z[seg][3] += a.w;
                                z[seg][4] += b.x; z[seg][5] += b.y; z[seg][6] += b.z; z[seg][7] += b.w;
                            }
                        }
                    }
                    if constexpr (GATED) {
#pragma unroll
                        for (int k = 0; k < 8; ++k) z[0][k] = activate<FORGE_ACT_SILU>(z[0][k]) * z[1][k];
                    } else {
#pragma unroll
                        for (int k = 0; k < 8; ++k) z[0][k] += s_bias[g * 8 + k];
                        activate_all(p.act, z[0]);
                        const uint32_t rw[4] = {r16.x, r16.y, r16.z, r16.w};
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            z[0][2 * k] += widen16<F16>(static_cast<uint16_t>(rw[k] & 0xffffu));
                            z[0][2 * k + 1] += widen16<F16>(static_cast<uint16_t>(rw[k] >> 16));
                        }
                    }
                    *reinterpret_cast<uint4*>(place(lane, i)) =
                        make_uint4(pack16<F16>(z[0][0], z[0][1]), pack16<F16>(z[0][2], z[0][3]),
                                   pack16<F16>(z[0][4], z[0][5]), pack16<F16>(z[0][6], z[0][7]));
                }
            }
            __syncwarp();
            if (ngroups > 0) {
                const int col0 = own0 + first * 8;
                uint16_t* y0 = p.y + (size_t)(m0 + quarter * 32) * p.N + col0;
                for (int it = 0; it < pieces; ++it) {
                    const int idx = it * 32 + lane, r = idx >> pieces_log2, c = idx & (pieces - 1);
                    if (m0 + quarter * 32 + r < p.M && col0 + c * 8 < p.N)
                        *reinterpret_cast<uint4*>(y0 + (size_t)r * p.N + c * 8) = *reinterpret_cast<const uint4*>(place(r, c));
                }
            }
        }
        __syncwarp();
    }
    // every thread of the cluster takes part in both phases of the cluster barrier
    if (S > 1 && !(warp >= 2 && warp < 2 + kEpiWarps)) {
        cluster_wait();
        cluster_arrive();
        cluster_wait();
    }

    if (failed) {
        atomicExch(p.status, 1);
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);  // let copies and MMAs in flight land
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, BN);
    }
}

constexpr int kSmemWhole = 224 * 1024, kSmemHalf = 110 * 1024;  // one or two CTAs per SM
constexpr int kBarBytes = (2 * kMaxStages + 2) * 8 + 128 * 4;

template <bool W_NK, bool F16, bool GATED>
int launch_split(const SplitPlan& plan, const void* x, const void* w, const void* w_up, const void* b, const void* residual,
                 void* y, int M, int N, int K, int act, cudaStream_t s) {
    const int bn = plan.bn, bno = GATED ? bn / 2 : bn, S = plan.split;
    SplitParams p;
    p.bias = static_cast<const uint16_t*>(b);
    p.residual = static_cast<const uint16_t*>(residual);
    p.y = static_cast<uint16_t*>(y);
    p.M = M; p.N = N; p.K = K;
    p.act = act;
    p.bn_log2 = __builtin_ctz(bn);
    p.split_log2 = __builtin_ctz(S);
    p.xrows = M >= kBM ? kBM : (M + 7) / 8 * 8;
    p.recv_rows = M >= kBM ? kBM : (M + 31) / 32 * 32;
    const int stage_bytes = p.xrows * kBK * 2 + bn * kBK * 2;
    const int recv_bytes = (S - 1) * (bn / S) * p.recv_rows * 4;
    const int kblocks = (K + kBK - 1) / kBK, nkb_max = (kblocks + S - 1) / S;
    int stages = ((plan.two_per_sm ? kSmemHalf : kSmemWhole) - recv_bytes - kBarBytes - 1024) / stage_bytes;
    if (stages > nkb_max) stages = nkb_max;
    if (stages > kMaxStages) stages = kMaxStages;
    if (stages < 2) stages = 2;  // the epilogue's staging rows take up to 32 KB of the ring
    p.stages = stages;
    p.recv_off = stages * stage_bytes;
    p.bar_off = p.recv_off + recv_bytes;
    int total = p.bar_off + kBarBytes;
    // an MMA reads 128 rows of A, also where the X tile is shorter
    if (total < (stages - 1) * stage_bytes + kABytes) total = (stages - 1) * stage_bytes + kABytes;
    total += 1024;  // slack to align the base
    const long long ctas = (long long)((M + kBM - 1) / kBM) * ((N + bno - 1) / bno) * S;
    if (ctas > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    p.prefetch = plan.two_per_sm || ctas * 2 <= sm_count();
    p.status = device_status_word();
    if (!p.status) return FORGE_ERR_CUDA;

    CUtensorMap tmap_x, tmap_w, tmap_w2;
    {
        const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M};
        const uint64_t strides[1] = {(uint64_t)K * 2};
        const uint32_t box[2] = {kBK, (uint32_t)p.xrows};
        if (!encode_tmap_bf16_sw128(&tmap_x, x, 2, dims, strides, box)) return FORGE_ERR_CUDA;
    }
    {
        const uint64_t dims[2] = {(uint64_t)(W_NK ? K : N), (uint64_t)(W_NK ? N : K)};
        const uint64_t strides[1] = {(uint64_t)(W_NK ? K : N) * 2};
        const uint32_t box[2] = {64, W_NK ? (uint32_t)bno : (uint32_t)kBK};
        if (!encode_tmap_bf16_sw128(&tmap_w, w, 2, dims, strides, box)) return FORGE_ERR_CUDA;
        if (GATED && !encode_tmap_bf16_sw128(&tmap_w2, w_up, 2, dims, strides, box)) return FORGE_ERR_CUDA;
    }
    if (!GATED) tmap_w2 = tmap_w;
    auto kernel = linear_split_kernel<W_NK, F16, GATED>;
    FORGE_SET_SMEM_ONCE(kernel, kSmemWhole);
    FORGE_CUDA_TRY(launch_pdl_cluster(kernel, dim3((unsigned)ctas), dim3(kThreads), total, S, s, tmap_x, tmap_w, tmap_w2, p));
    return finish_launch(1);
}

}  // namespace

// One row tile (M <= 128).  Up to 64 rows, 64-column tiles at two CTAs per SM; above, where a stage is mostly X, one
// per SM.  S grows while all CTAs still run at once (a little under two / one per SM: clusters of eight do not tile
// every GPC) and each keeps two / three k-blocks to itself (below that the exchange costs more than the shorter loop
// saves: 1 x 768 x 768 4.2 us with S = 4, 4.4 us with S = 8; 128 x 2304 x 768 5.5 us with S = 2, 6.3 us with S = 4).
// Wider outputs take 128-column tiles (16 x 32768 x 4096: 44.3 us, 47.3 us with 64 columns).
SplitPlan linear_split_plan_row(bool gated, int M, int N, int K, int sms) {
    const int kblocks = (K + kBK - 1) / kBK;
    const bool narrow = M <= 64;
    SplitPlan pl;
    pl.two_per_sm = narrow && !gated;
    const long long room = pl.two_per_sm ? 2LL * sms * 8 / 9 : (long long)sms * 8 / 9;
    // gated: a 128-column accumulator is 64 output columns
    pl.bn = gated ? 128 : 64;
    const long long tiles64 = (N + 63) / 64;
    if (tiles64 > room && !gated) pl.bn = 128;
    const int bno = gated ? pl.bn / 2 : pl.bn;
    const long long tiles = (N + bno - 1) / bno;
    if (tiles > room) pl.two_per_sm = true;  // several rounds: the next tile's copies overlap the last one's epilogue
    pl.split = 1;
    while (pl.split < 8 && tiles * pl.split * 2 <= room && kblocks >= pl.split * 2 * (narrow ? 2 : 3)) pl.split *= 2;
    return pl;
}

// Several row tiles: the split kernel against CTA pairs, by estimated microseconds: fixed cost of launch, first copy, epilogue
// and exchange, plus the time of a k-block.  A 128 x 128 tile is bound by shared memory (64 KB written and read per k-block,
// up to 0.28 us for 0.13 us of tensor core), a pair's 256 x 256 tile is not (0.285 us for four times the work), but a quarter as many
// tiles leave SMs idle.  The estimates rank the plans, they do not predict times (up to a third too long for one CTA
// per tile and long K, a quarter too short for many rounds of pairs): of 22 shapes of 130-4342 rows, 256-14336 columns and K
// 136-14336, measured with every plan, the plan taken was the fastest or within 3 % of it (256 x 4096 x 14336 35.5 us, pairs 72.5;
// 596 x 3072 x 768 8.9 and 9.7; 458 x 8192 x 2048 pairs; profiles/linear_plan_rows.md has them all).
bool linear_split_plan_rows(int M, int N, int K, int sms, SplitPlan* plan) {
    const int kblocks = (K + kBK - 1) / kBK;
    const long long t2 = (long long)((M + 255) / 256) * ((N + 255) / 256), pairs = sms / 2;
    *plan = {128, 1, true};
    double best = 1e30;
    bool split = pairs < 1;
    if (!split) {
        const long long rem = t2 % pairs;
        const double rounds = (double)(t2 / pairs) + (rem == 0 ? 0.0 : 2 * rem <= pairs && t2 > pairs ? 0.55 : 1.0);
        best = 6.7 + 0.285 * rounds * kblocks;
    }
    const long long tiles_m = (M + kBM - 1) / kBM;
    for (int bn = 64; bn <= 128; bn *= 2) {
        const long long tiles = tiles_m * ((N + bn - 1) / bn);
        for (int S = 1; S <= 8 && S <= kblocks; S *= 2) {
            if (tiles * S > (S == 1 ? sms : sms * 8 / 9)) break;
            const double t = 4.9 + (bn == 64 ? 0.18 : 0.28) * ((kblocks + S - 1) / S) + (S == 1 ? 0.0 : bn == 64 ? 0.8 : 1.3);
            if (t < best) { best = t; split = true; *plan = {bn, S, false}; }
        }
    }
    return split;
}

int linear_split(const SplitPlan& plan, bool f16, const void* x, const void* w, const void* b, const void* residual, void* y,
                 int M, int N, int K, int act, int w_layout, cudaStream_t s) {
    if (f16)
        return w_layout == FORGE_W_NK ? launch_split<true, true, false>(plan, x, w, nullptr, b, residual, y, M, N, K, act, s)
                                      : launch_split<false, true, false>(plan, x, w, nullptr, b, residual, y, M, N, K, act, s);
    return w_layout == FORGE_W_NK ? launch_split<true, false, false>(plan, x, w, nullptr, b, residual, y, M, N, K, act, s)
                                  : launch_split<false, false, false>(plan, x, w, nullptr, b, residual, y, M, N, K, act, s);
}

int linear_split_swiglu(const SplitPlan& plan, const void* x, const void* w_gate, const void* w_up, void* y, int M, int N,
                        int K, int w_layout, cudaStream_t s) {
    return w_layout == FORGE_W_NK
               ? launch_split<true, false, true>(plan, x, w_gate, w_up, nullptr, nullptr, y, M, N, K, FORGE_ACT_NONE, s)
               : launch_split<false, false, true>(plan, x, w_gate, w_up, nullptr, nullptr, y, M, N, K, FORGE_ACT_NONE, s);
}

}  // namespace forge
