// Weight-only int8 linear (fp16 activations, int8 weights [N,K] with one fp32 scale per output channel, the
// W-int8 / A-fp16 setting of the paper's largest model): Y = act(X W^T * scale + b) + residual.
//
// The product is computed transposed: D[feature, token] = Wq[feature, :] . X[token, :], with the weights as the A operand
// in TENSOR MEMORY and the tokens as the B operand.  The int8 tile arrives by TMA, converter threads (thread = feature
// = TMEM lane) widen their row to fp16 and write it to tensor memory, where the tensor core reads it.
// The widening is exact: bytes (u, 0x64) read as fp16 are 1024 + u with u = w + 128, minus 1152; the scale factors out
// of the sum over K and multiplies the fp32 accumulator.
//
// What bounds it: an SM takes in at most 64 bytes a cycle, and a 64-deep k-block of 128 features brings 8 KB of int8 and
// 128 bytes per token; the widened operand no longer passes through shared memory twice, and the X tile has the tokens
// that exist instead of 128 rows.  Weights cold, against the one-CTA kernel with the fp16 operand in shared memory:
//   1 x 14336 x 4096 40 -> 16 us, 128 x 14336 x 4096 41 -> 22 us, 16 x 4096 x 14336 120 -> 15 us,
//   300 x 4096 x 14336 120 -> 41 us, 8192 x 8192 x 4096 504 -> 454 us (1210 TFLOP/s).
// 128-deep stages (rows of 128 bytes) were slower (20.7 and 25.8 us for the first two); more than one A operand per
// converter group changes nothing.
//
// Tokens per tile (nt): all of them up to 192, else M in equal shares of at most 192 (a multiple of 16): 300 tokens
// are two tiles of 160, not three of 128.  Two accumulators of 192 columns: the epilogue of a tile overlaps the k-loop of
// the next (persistent CTAs).  Outputs with few tiles split K over clusters as linear_split.cu does: CTA r of S sums
// its share of the k-blocks, owns a share of the tokens, and is sent the others' partial sums through shared memory.
//
// A cluster's CTAs wait for one another, so two clusters must not each hold tensor memory that the other one's CTAs wait for.
// Beside one of these CTAs (832 threads of 72 registers, all 512 columns) an SM has 5600 registers left, and the CTAs of the other
// kernels that run in clusters (linear_pair.cu, linear_split.cu) take 23000 and more.
//
// Warps: 0 TMA producer, 1 MMA issuer and TMEM owner, then six quads of four warps (128 TMEM lanes): epilogue quads, which
// take groups of tokens in turn, and three or four converter quads ("groups"), which take k-blocks in turn, each with its
// own A operand.
#include <cuda_fp16.h>

#include "activations.cuh"
#include "forge_common.cuh"
#include "linear_w8.cuh"
#include "sm100_ptx.cuh"
#include "tmap.cuh"

namespace forge {
namespace {

using namespace ptx;

constexpr int kBF = 128;            // features per tile
constexpr int kBK = 64;
constexpr int kMaxTokens = 192;     // tokens per tile
constexpr int kWarpQuads = 6;       // epilogue warps and converter groups, in units of four warps (128 TMEM lanes)
constexpr int kThreads = 64 + kWarpQuads * 128;
constexpr int kMaxGroups = 4;
constexpr int kMaxEpiWarps = 16;
constexpr int kColA = 2 * kMaxTokens;  // TMEM: accumulators at 0 and 192, A operands (32 columns per group) from 384
constexpr int kTmemCols = 512;
constexpr int kMaxStages = 16;
constexpr int kSmemMax = 224 * 1024;
constexpr int kOutBytes = kMaxEpiWarps * 1024;
constexpr int kBarBytes = (2 * kMaxStages + 2 * kMaxGroups + 4 + 1) * 8;

struct W8Params {
    const uint16_t* bias;
    const uint16_t* residual;  // may be y
    const float* scale;
    uint16_t* y;
    int M, N, K;
    int act;
    int nt, tiles_t;     // tokens per tile, token tiles
    int split_log2;      // CTAs per tile
    int own4;            // 4-token pieces a CTA of a cluster finishes
    int stages;          // at least as many as converter groups
    int recv_off, out_off, bar_off;  // byte offsets in shared memory
    int* status;
};

__device__ __forceinline__ uint32_t widen2(uint32_t bits, __half2 off) {
    const __half2 h = __hsub2(*reinterpret_cast<__half2*>(&bits), off);
    return *reinterpret_cast<const uint32_t*>(&h);
}

template <int kGroups>
__global__ void __launch_bounds__(kThreads, 1)
linear_w8_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w, const W8Params p) {
    constexpr int kEpiQuads = kWarpQuads - kGroups, kEpiWarps = 4 * kEpiQuads;
    extern __shared__ uint8_t smem_raw[];
    // the same offset in every CTA of the cluster (dynamic shared memory starts at the same address in each)
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + p.bar_off);
    uint64_t* empty = full + kMaxStages;
    uint64_t* conv_full = empty + kMaxStages;
    uint64_t* conv_empty = conv_full + kGroups;
    uint64_t* tmem_full = conv_empty + kGroups;
    uint64_t* tmem_empty = tmem_full + 2;
    uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(tmem_empty + 2);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = 1 << p.split_log2;
    const int rank = (int)blockIdx.x & (S - 1);
    const int first_tile = (int)blockIdx.x >> p.split_log2, tile_step = (int)gridDim.x >> p.split_log2;
    const int num_tiles = p.tiles_t * ((p.N + kBF - 1) / kBF);
    const int kblocks = (p.K + kBK - 1) / kBK;
    const int kb0 = (int)((long long)kblocks * rank >> p.split_log2);
    const int nkb = (int)((long long)kblocks * (rank + 1) >> p.split_log2) - kb0;
    constexpr int kRawBytes = kBF * kBK;
    const int stage_bytes = kRawBytes + p.nt * (kBK * 2);  // int8 rows, then X
    // tiles of the same features follow one another: their weights are still in L2
    auto feature0 = [&](int tile) { return tile / p.tiles_t * kBF; };
    auto token0 = [&](int tile) { return tile % p.tiles_t * p.nt; };

    if (threadIdx.x == 0) {
        for (int i = 0; i < p.stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
        for (int i = 0; i < kGroups; ++i) { mbar_init(&conv_full[i], 4); mbar_init(&conv_empty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&tmem_full[i], 1); mbar_init(&tmem_empty[i], kEpiWarps); }
        fence_mbar_init();
        prefetch_tmap(&tmap_w);
        prefetch_tmap(&tmap_x);
    }
    if (warp == 1) {
        tmem_alloc(tmem_base_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_base_slot;
    bool failed = false;
    if (S > 1) cluster_arrive();  // this CTA runs: its shared memory may be written (awaited before the exchange)
    pdl_launch_dependents();
    pdl_wait();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int stage = 0;
            uint32_t phase = 0;
            for (int tile = first_tile; tile < num_tiles && !failed; tile += tile_step) {
                const int f0 = feature0(tile), t0 = token0(tile);
                for (int kb = kb0; kb < kb0 + nkb; ++kb) {
                    if (!mbar_wait_relaxed(&empty[stage], phase ^ 1)) { failed = true; break; }
                    uint8_t* raw = smem + stage * stage_bytes;
                    mbar_expect_tx(&full[stage], stage_bytes);
                    tma_load_2d(raw, &tmap_w, &full[stage], kb * kBK, f0);
                    tma_load_2d(raw + kRawBytes, &tmap_x, &full[stage], kb * kBK, t0);
                    if (++stage == p.stages) { stage = 0; phase ^= 1; }
                }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idesc = make_idesc_f16(kBF, p.nt, /*a_mn_major=*/false, /*b_mn_major=*/false);
            int stage = 0, grp = 0, it = 0;
            uint32_t gphase = 0;
            for (int tile = first_tile; tile < num_tiles && !failed; tile += tile_step, ++it) {
                const int acc = it & 1;
                if (!mbar_wait(&tmem_empty[acc], ((it >> 1) & 1) ^ 1)) { failed = true; break; }
                tc_fence_after_sync();
                const uint32_t d_tmem = tmem_base + acc * kMaxTokens;
                for (int kb = 0; kb < nkb; ++kb) {
                    // the converters have seen the stage's barrier complete: X has landed too
                    if (!mbar_wait(&conv_full[grp], gphase)) { failed = true; break; }
                    tc_fence_after_sync();
                    const uint32_t a_tmem = tmem_base + kColA + grp * (kBK / 2);
                    const uint64_t b_desc = make_smem_desc(smem_u32(smem + stage * stage_bytes + kRawBytes), 16, 1024);
#pragma unroll
                    for (int k = 0; k < kBK / 16; ++k)
                        mma_ts(d_tmem, a_tmem + k * 8, b_desc + k * (32 >> 4), idesc, (kb | k) != 0);
                    mma_commit(&conv_empty[grp]);
                    mma_commit(&empty[stage]);
                    if (++grp == kGroups) { grp = 0; gphase ^= 1; }
                    if (++stage == p.stages) stage = 0;
                }
                if (failed) break;
                mma_commit(&tmem_full[acc]);
            }
        }
        __syncwarp();
    } else if (warp >= 2 + kEpiWarps) {
        // ------------------------------------------------------------------ int8 -> fp16 converters
        const int group = (warp - 2 - kEpiWarps) >> 2, quarter = warp & 3;
        const int row = quarter * 32 + lane;
        const uint32_t a_tmem = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + kColA + group * (kBK / 2);
        const __half2 off = __floats2half2_rn(1152.f, 1152.f);
        int stage = group;
        uint32_t phase = 0, gphase = 0;
        int tiles = 0;
        for (int tile = first_tile; tile < num_tiles; tile += tile_step) ++tiles;
        const int total = tiles * nkb;  // k-blocks of this CTA over all its tiles
        for (int g = group; g < total; g += kGroups) {
            // First that the tensor core has read this group's previous operand: with at least kGroups stages the barrier of
            // the int8 tile is then at most one phase behind, and its parity means what is asked.
            if (!warp_wait_relaxed(&conv_empty[group], gphase ^ 1) || !warp_wait(&full[stage], phase)) { failed = true; break; }
            gphase ^= 1;
            const uint8_t* raw = smem + stage * stage_bytes + row * kBK;
            uint4 in[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) in[c] = *reinterpret_cast<const uint4*>(raw + ((c ^ ((row >> 1) & 3)) << 4));
            uint32_t o[32];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const uint32_t wds[4] = {in[c].x ^ 0x80808080u, in[c].y ^ 0x80808080u, in[c].z ^ 0x80808080u, in[c].w ^ 0x80808080u};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    o[c * 8 + 2 * j] = widen2(__byte_perm(wds[j], 0x64646464u, 0x4140), off);
                    o[c * 8 + 2 * j + 1] = widen2(__byte_perm(wds[j], 0x64646464u, 0x4342), off);
                }
            }
            tc_fence_after_sync();
            tmem_st_x32(a_tmem, o);
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&conv_full[group]);
            if ((stage += kGroups) >= p.stages) { stage -= p.stages; phase ^= 1; }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ epilogue
        const int quarter = warp & 3;       // TMEM lane quarter this warp may access
        const int share = (warp - 2) >> 2;  // takes every kEpiQuads-th group of tokens
        const int frow = quarter * 32 + lane;
        uint8_t* rows = smem + p.out_off + (warp - 2) * 1024;  // up to 16 tokens x 32 features of this warp
        // The T tokens of z from `token` of the warp's 32 features: scale, bias, activation, residual, rounding.  A thread holds one
        // feature; the rows go through shared memory so that they are read and written in pieces of 16 bytes (2-byte
        // accesses made the epilogue of a 768-deep product longer than its k-loop: 4000 x 3072 x 768 43 us).
        auto finish = [&](auto& z, int col0, float sc, float bi, int token, int tokens_end) {
            constexpr int T = sizeof(z) / sizeof(float);
            const int piece_col = col0 + (lane & 3) * 8;
            constexpr int kPieces = (T + 7) / 8;
            auto for_pieces = [&](auto f) {
#pragma unroll
                for (int i = 0; i < kPieces; ++i) {
                    const int t = i * 8 + (lane >> 2);
                    if (t < T && token + t < tokens_end && piece_col < p.N)
                        f(i, (size_t)(token + t) * p.N + piece_col, reinterpret_cast<uint4*>(rows + t * 64 + (lane & 3) * 16));
                }
            };
            uint4 res[kPieces];  // on its way while the activation is computed
            if (p.residual != nullptr)
                for_pieces([&](int i, size_t at, uint4*) { res[i] = *reinterpret_cast<const uint4*>(p.residual + at); });
#pragma unroll
            for (int k = 0; k < T; ++k) z[k] = fmaf(z[k], sc, bi);
            activate_all(p.act, z);
            if (p.residual != nullptr) {
                for_pieces([&](int i, size_t, uint4* r) { *r = res[i]; });
                __syncwarp();
#pragma unroll
                for (int k = 0; k < T; ++k) z[k] += __half2float(*reinterpret_cast<const __half*>(rows + k * 64 + lane * 2));
                __syncwarp();
            }
#pragma unroll
            for (int k = 0; k < T; ++k) *reinterpret_cast<__half*>(rows + k * 64 + lane * 2) = __float2half_rn(z[k]);
            __syncwarp();
            for_pieces([&](int, size_t at, uint4* r) { *reinterpret_cast<uint4*>(p.y + at) = *r; });
            __syncwarp();
        };
        int it = 0;
        for (int tile = first_tile; tile < num_tiles; tile += tile_step, ++it) {
            const int acc = it & 1;
            const int feature = feature0(tile) + frow, t0 = token0(tile);
            const int col0 = feature - lane;
            const int tokens_end = min(t0 + p.nt, p.M), ntok = tokens_end - t0;
            const bool f_ok = feature < p.N;
            const float sc = f_ok ? p.scale[feature] : 0.f;
            const float bi = f_ok && p.bias != nullptr ? __half2float(__ushort_as_half(p.bias[feature])) : 0.f;
            if (!warp_wait(&tmem_full[acc], (it >> 1) & 1)) { failed = true; break; }
            tc_fence_after_sync();
            const uint32_t taddr = tmem_base + acc * kMaxTokens + (static_cast<uint32_t>(quarter * 32) << 16);
            if (S == 1) {
#pragma unroll 1
                for (int c = share * 16; c < ntok; c += kEpiQuads * 16) {
                    uint32_t r[16];
                    tmem_ld_x16(taddr + c, r);
                    tmem_ld_wait();
                    float z[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) z[k] = __uint_as_float(r[k]);
                    finish(z, col0, sc, bi, t0 + c, tokens_end);
                }
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tmem_empty[acc]);
            } else {
                // one tile per cluster.  recv of an owner: [source slot][4-token piece][feature] of 16 bytes
                uint8_t* recv = smem + p.recv_off;
                const uint32_t recv0 = smem_u32(recv);
                const int pieces = (ntok + 3) >> 2;
                const int own_begin = rank * p.own4, own_end = min(own_begin + p.own4, pieces);
                cluster_wait();  // every CTA of the cluster runs
#pragma unroll 1
                for (int c = share * 4; c < pieces; c += kEpiQuads * 4) {
                    uint32_t r[16];
                    tmem_ld_x16(taddr + c * 4, r);
                    tmem_ld_wait();
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int piece = c + q, owner = piece / p.own4;
                        if (owner == rank || piece >= pieces) continue;
                        const int slot = rank - (rank > owner ? 1 : 0);
                        const uint32_t at = (uint32_t)((slot * p.own4 + piece - owner * p.own4) * kBF + frow) * 16;
                        st_cluster_v4(map_addr_to_cta(recv0 + at, owner), r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
                    }
                }
                cluster_arrive();
                cluster_wait();  // the other CTAs' partial sums have arrived
#pragma unroll 1
                for (int piece = own_begin + share; piece < own_end; piece += kEpiQuads) {
                    uint32_t mine[4];
                    tmem_ld_x4(taddr + piece * 4, mine);
                    tmem_ld_wait();
                    float z[4] = {0.f, 0.f, 0.f, 0.f};
                    for (int src = 0; src < S; ++src) {  // in rank order: results do not depend on timing
                        if (src == rank) {
#pragma unroll
                            for (int k = 0; k < 4; ++k) z[k] += __uint_as_float(mine[k]);
                        } else {
                            const int slot = src - (src > rank ? 1 : 0);
                            const float4 a = *reinterpret_cast<const float4*>(
                                recv + (size_t)((slot * p.own4 + piece - own_begin) * kBF + frow) * 16);
                            z[0] += a.x; z[1] += a.y; z[2] += a.z; z[3] += a.w;
                        }
                    }
                    finish(z, col0, sc, bi, t0 + piece * 4, tokens_end);
                }
            }
        }
        if (S > 1 && failed) { cluster_wait(); cluster_arrive(); cluster_wait(); }  // the one tile's barriers were not reached
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
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

template <int kGroups>
int launch_w8(const CUtensorMap& tmap_x, const CUtensorMap& tmap_w, const W8Params& p, unsigned grid, int smem_bytes, int S,
              cudaStream_t s) {
    FORGE_SET_SMEM_ONCE(linear_w8_kernel<kGroups>, kSmemMax);
    FORGE_CUDA_TRY(launch_pdl_cluster(linear_w8_kernel<kGroups>, dim3(grid), dim3(kThreads), smem_bytes, S, s, tmap_x, tmap_w, p));
    return finish_launch(1);
}

}  // namespace

bool linear_w8_plan(int M, int N, int K, int sms, W8Plan* plan) {
    W8Plan& pl = *plan;
    const int kblocks = (K + kBK - 1) / kBK;
    const long long tiles_f = (N + kBF - 1) / kBF;
    pl.tiles_t = (M + kMaxTokens - 1) / kMaxTokens;
    pl.nt = ((M + pl.tiles_t - 1) / pl.tiles_t + 15) / 16 * 16;
    if (pl.tiles_t * tiles_f > sms) {  // several rounds: the smallest tiles that need no more of them
        const long long rounds = (pl.tiles_t * tiles_f + sms - 1) / sms, most = rounds * sms / tiles_f;
        pl.nt = (int)((M + most - 1) / most + 15) / 16 * 16;
        pl.tiles_t = (M + pl.nt - 1) / pl.nt;
    }
    pl.tiles = pl.tiles_t * tiles_f;
    // Long k-loops in several rounds keep the converters busy: four groups (8192 x 8192 x 4096 454 us, 507 with three).
    // Everything else gains more from a third quad of epilogue warps (8192 x 768 x 768 16.7 against 24.6 us, with erf and
    // residual 30 against 42; 400 x 3072 x 768 9.0 against 9.6), and a single token does not notice (16.0 both).
    pl.groups = pl.tiles > sms && kblocks >= 48 ? 4 : 3;
    // as many CTAs per tile as run at once (clusters of eight do not tile every GPC) with two k-blocks or more each
    // (1 x 768 x 768: 4.0 us, with three or more 4.6 us)
    pl.split = 1;
    while (pl.split < 8 && pl.tiles * pl.split * 2 <= sms * 8 / 9 && kblocks >= pl.split * 2 * 2) pl.split *= 2;
    const int stage_bytes = kBF * kBK + pl.nt * kBK * 2;  // at most 32 KB
    for (;; pl.split /= 2) {
        pl.own4 = pl.split > 1 ? (pl.nt / 4 + pl.split - 1) / pl.split : 0;
        pl.recv_bytes = (pl.split - 1) * pl.own4 * kBF * 16;  // at most 84 KB (192 tokens, S = 8)
        pl.stages = (kSmemMax - pl.recv_bytes - kOutBytes - kBarBytes - 1024) / stage_bytes;
        if (pl.stages > kMaxStages) pl.stages = kMaxStages;
        // The converters need a stage per group (their barrier parities, linear_w8_kernel).  192 tokens and S = 8 leave three
        // stages for three groups; with S = 1 there are six and more.
        if (pl.stages >= pl.groups || pl.split == 1) break;
    }
    return pl.tiles <= 2147483647LL && pl.stages >= pl.groups;
}

int linear_w8(const void* x, const void* w_int8, const float* scale, const void* b, const void* residual, void* y, int M,
              int N, int K, int act, cudaStream_t s) {
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    W8Plan pl;
    if (!linear_w8_plan(M, N, K, sms, &pl)) return FORGE_ERR_UNSUPPORTED;
    W8Params p;
    p.bias = static_cast<const uint16_t*>(b);
    p.residual = static_cast<const uint16_t*>(residual);
    p.scale = scale;
    p.y = static_cast<uint16_t*>(y);
    p.M = M; p.N = N; p.K = K;
    p.act = act;
    p.nt = pl.nt;
    p.tiles_t = pl.tiles_t;
    p.split_log2 = __builtin_ctz(pl.split);
    p.own4 = pl.own4;
    p.stages = pl.stages;
    p.recv_off = pl.stages * (kBF * kBK + pl.nt * kBK * 2);
    p.out_off = p.recv_off + pl.recv_bytes;
    p.bar_off = p.out_off + kOutBytes;
    const int total = p.bar_off + kBarBytes + 1024;
    p.status = device_status_word();
    if (!p.status) return FORGE_ERR_CUDA;
    CUtensorMap tmap_x, tmap_w;
    {
        const uint64_t dims[2] = {(uint64_t)K, (uint64_t)M};
        const uint64_t strides[1] = {(uint64_t)K * 2};
        const uint32_t box[2] = {kBK, (uint32_t)p.nt};
        if (!encode_tmap_bf16_sw128(&tmap_x, x, 2, dims, strides, box)) return FORGE_ERR_CUDA;
    }
    {
        const uint64_t dims[2] = {(uint64_t)K, (uint64_t)N};
        const uint64_t strides[1] = {(uint64_t)K};
        const uint32_t box[2] = {kBK, kBF};
        if (!encode_tmap_u8_sw64(&tmap_w, w_int8, 2, dims, strides, box)) return FORGE_ERR_CUDA;
    }
    const long long grid = pl.split > 1 ? pl.tiles * pl.split : (pl.tiles < sms ? pl.tiles : sms);
    return pl.groups == 4 ? launch_w8<4>(tmap_x, tmap_w, p, (unsigned)grid, total, pl.split, s)
                          : launch_w8<3>(tmap_x, tmap_w, p, (unsigned)grid, total, pl.split, s);
}

}  // namespace forge
