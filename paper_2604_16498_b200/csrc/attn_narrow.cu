// Fused attention for head sizes up to 64 (Eq. 8 / Eq. 9, the same operator as attn_bf16.cu, without an additive bias; many short tiles
// run there: many_short_tiles()).
//
// With 64 columns of output a 64-key step is 256 cycles of tensor core against 512 of the special-function unit's exponentials, and
// the rest of a step (barriers, tensor-memory round trips, fences) is as long as both.  So the kernel is small and the SM
// holds three of its CTAs: one query tile of 128 rows each, 160 threads, 65 KB of shared memory and 160 tensor-memory columns.
// While one tile waits, the others keep the special-function unit busy, and the hardware scheduler hands out the tiles, longest
// first.
//
//   tensor memory   S at column 0 (64 fp32 columns), O at 64; P (16-bit, two per column) in 32 columns of an allocation of its own,
//                   from where it is the A operand of P V
//   shared memory   Q 16 KB (the output is staged in its place), three stages of 64 keys for K and three for V, 8 KB each
//   warps 0-3       softmax, rescale and epilogue: thread = tile row = TMEM lane
//   warp 4          one lane issues the copies and the MMAs; the warp owns the TMEM allocations
// Per step g: S(g) complete -> the softmax warps read it into registers -> S(g + 1) = Q K(g + 1)^T is issued into the same columns and
// runs beside the exponentials of step g -> P(g) stored -> O += P(g) V(g).  P(g) may be stored once the product of step g - 1 has
// read P(g - 1); with P over S instead, the next scores waited for this step's product, and four CTAs per SM took 870 cycles per
// tile and step.
// O is rescaled in tensor memory only when a row's maximum grows by more than 2^8 (the stale maximum is kept otherwise; the final
// division by l uses the same reference).
#include "attn_math.cuh"
#include "attn_narrow.cuh"
#include "attn_tiles.cuh"
#include "forge_common.cuh"
#include "sm100_ptx.cuh"
#include "tmap.cuh"

#include <type_traits>

namespace forge {
namespace {

using namespace ptx;

constexpr int kD = 64;            // the kernel's head dimension
constexpr int kBM = 128;          // rows of a tile
constexpr int kStep = 64;         // keys per step and per K/V stage
constexpr int kThreads = 160;
constexpr int kCtasPerSm = 3;
constexpr int kStages = 3;        // of K and of V
constexpr int kTmemCols = 128;    // S and O
constexpr int kTmemColsP = 32;
constexpr int kColO = 64;
// of the 32 score pairs of an unmasked step, how many take their exponentials on the FMA pipe (0 / 4 / 8 / 12: 4 x 16 heads x 2048 not
// causal 97.9 / 97.0 / 95.1 / 97.6 us)
constexpr int kFmaExpPairs = 8;
constexpr float kRescaleThreshold = 8.0f;  // log2 units

struct NarrowSmem {
    static constexpr int kQBytes = kBM * 128;
    static constexpr int kKVBytes = kStep * 128;
    static constexpr int kKOff = kQBytes;
    static constexpr int kVOff = kKOff + kStages * kKVBytes;
    static constexpr int kBarOff = kVOff + kStages * kKVBytes;
    static constexpr int kNumBars = 6 + 2 * kStages;  // q_full, k_full[3], v_full[3], s_full, s_read, p_ready, pv_done, o_staged
    static constexpr int kTotal = kBarOff + kNumBars * 8 + 16;
    static constexpr int kAlloc = kTotal + 1024;
};

struct NarrowParams {
    uint16_t* out;
    long long o_sb, o_sh, o_ss;  // element strides of out between batch entries, heads and rows
    const int32_t* lens;
    int B, Hq, Hkv, Sq, Skv, head_dim, mask_kind;
    int pack, head_rows;  // query heads in a tile and the rows of each (attn_tiles.cuh)
    float scale_log2;     // > 0
    int* status;
};

template <bool F16>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
attn_narrow_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                   const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_o,
                   const NarrowParams p) {
    using L = NarrowSmem;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem;
    uint8_t* sK = smem + L::kKOff;
    uint8_t* sV = smem + L::kVOff;
    uint64_t* q_full = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint64_t* k_full = q_full + 1;         // [3] step g uses stage g % 3
    uint64_t* v_full = k_full + kStages;   // [3]
    uint64_t* s_full = v_full + kStages;   // S(g) is complete
    uint64_t* s_read = s_full + 1;         // S(g) is in the softmax threads' registers
    uint64_t* p_ready = s_read + 1;
    uint64_t* pv_done = p_ready + 1;       // O holds the product of step g
    uint64_t* o_staged = pv_done + 1;      // all four warps' rows of the output lie in Q's place
    uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(o_staged + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int causal_off = p.Skv - p.Sq;
    const bool causal = (p.mask_kind & FORGE_MASK_CAUSAL) != 0, padding = (p.mask_kind & FORGE_MASK_PADDING) != 0;
    // tiles longest first (causal): the last rows of every head group, then the ones before, ...
    const int groups = p.Hq / p.pack, heads = p.B * groups, q_tiles = (int)gridDim.x / heads;
    const int round = (int)blockIdx.x / heads, bg = (int)blockIdx.x - round * heads;
    const int b = bg / groups, head = (bg - b * groups) * p.pack, kvh = head / (p.Hq / p.Hkv);
    const int q0 = (q_tiles - 1 - round) * p.head_rows;

    int kvlen = p.Skv, n = 0;  // n: steps visible to at least one row of the tile
    auto measure = [&]() {
        if (padding) kvlen = min(max(p.lens[b], 0), p.Skv);
        const int kv_end = max(causal ? min(kvlen, min(q0 + p.head_rows, p.Sq) + causal_off) : kvlen, 0);
        n = (kv_end + kStep - 1) / kStep;
    };
    const int rows = p.pack * p.head_rows;
    auto load = [&](const CUtensorMap* map, uint8_t* ring, uint64_t* full, int g) {
        if (g >= n) return;
        const int st = g % kStages;
        mbar_expect_tx(&full[st], L::kKVBytes);
        tma_load_4d(ring + st * L::kKVBytes, map, &full[st], 0, g * kStep, kvh, b);
    };
    // The first copies leave before the CTA's other threads are ready: their latency covers the rest of the set-up.  (The next kernel
    // may move in once every CTA has its tensor memory.)
    bool control = false;
    if (warp == 4) {
        // the small one first: after the other, it may land in the block that the next CTA's 128 columns need, and an SM holds two CTAs
        // for a while (8 x 12 x 1024 causal 31.5 -> 28.2 us, 2 x 12 x 4000 84 -> 73)
        tmem_alloc(tmem_base_slot + 1, kTmemColsP);
        tmem_alloc(tmem_base_slot, kTmemCols);
        tmem_relinquish();
        if (elect_one()) {
            control = true;
            prefetch_tmap(&tmap_q); prefetch_tmap(&tmap_k); prefetch_tmap(&tmap_v); prefetch_tmap(&tmap_o);
            mbar_init(q_full, 1);
            for (int i = 0; i < kStages; ++i) { mbar_init(&k_full[i], 1); mbar_init(&v_full[i], 1); }
            mbar_init(s_full, 1); mbar_init(s_read, 4); mbar_init(p_ready, 4); mbar_init(pv_done, 1); mbar_init(o_staged, 4);
            fence_mbar_init();
            fence_proxy_async_smem();
            pdl_launch_dependents();
            pdl_wait();
            measure();
            if (n > 0) {
                // rows beyond Sq and columns beyond head_dim are zero-filled by the TMA unit
                mbar_expect_tx(q_full, (uint32_t)rows * 128);
                tma_load_4d(sQ, &tmap_q, q_full, 0, q0, head, b);
                for (int g = 0; g < kStages; ++g) {
                    load(&tmap_k, sK, k_full, g);
                    load(&tmap_v, sV, v_full, g);
                }
            }
        }
        __syncwarp();
    }
    // Rows of the Q tile that are not in use are never written by the copy: zero scores, not whatever lies there.
    if (rows < kBM) {
        for (int i = rows * 8 + (int)threadIdx.x; i < kBM * 8; i += kThreads) reinterpret_cast<uint4*>(sQ)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = tmem_base_slot[0], tmem_p = tmem_base_slot[1];
    bool failed = false;
    pdl_wait();
    if (!control) measure();

    if (warp == 4) {
        // ------------------------------------------------------------------ copies and MMAs
        if (elect_one() && n > 0) {
            constexpr uint32_t idesc_s = F16 ? make_idesc_f16(kBM, kStep, false, false) : make_idesc_bf16(kBM, kStep, false, false);
            constexpr uint32_t idesc_o = F16 ? make_idesc_f16(kBM, kD, false, true) : make_idesc_bf16(kBM, kD, false, true);
            const uint64_t qd = make_smem_desc(smem_u32(sQ), 16, 1024);
            auto landed = [&](uint64_t* full, int g) { return mbar_wait(&full[g % kStages], (g / kStages) & 1); };
            auto issue_qk = [&](int g) {
                tc_fence_after_sync();
                const uint64_t kd = make_smem_desc(smem_u32(sK) + (g % kStages) * L::kKVBytes, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < kD / 16; ++kk) mma_ss(tmem_base, qd + kk * (32 >> 4), kd + kk * (32 >> 4), idesc_s, kk != 0);
                mma_commit(s_full);
            };
            if (!mbar_wait(q_full, 0) || !landed(k_full, 0)) failed = true;
            if (!failed) issue_qk(0);
            for (int g = 0; g < n && !failed; ++g) {
                // operands before the softmax warps' arrivals: then the MMAs go out at once
                if (g + 1 < n && !landed(k_full, g + 1)) { failed = true; break; }
                if (!mbar_wait(s_read, g & 1)) { failed = true; break; }
                if (g + 1 < n) issue_qk(g + 1);
                load(&tmap_k, sK, k_full, g + kStages);  // S(g) was complete: its K tile has been read
                if (!landed(v_full, g) || !mbar_wait(p_ready, g & 1)) { failed = true; break; }
                tc_fence_after_sync();
                // P: 16 keys = 8 columns of packed pairs.  V: MN-major, 16 keys = two 1024-byte groups (2048 bytes per MMA).
                const uint64_t vd = make_smem_desc(smem_u32(sV) + (g % kStages) * L::kKVBytes, L::kKVBytes, 1024);
#pragma unroll
                for (int kk = 0; kk < kStep / 16; ++kk)
                    mma_ts(tmem_base + kColO, tmem_p + kk * 8, vd + kk * (2048 >> 4), idesc_o, (g | kk) != 0);
                mma_commit(pv_done);
                if (g > 0) load(&tmap_v, sV, v_full, g - 1 + kStages);  // P(g) was stored after product g - 1: its V tile has been read
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------------ softmax / rescale / epilogue
        const int row = warp * 32 + lane;
        // head and query row within the tile; a row that is not in use goes along as the last head's first with Q = 0
        const bool live = row < rows;
        const int row_h = min(row / p.head_rows, p.pack - 1), qi = q0 + (live ? row - row_h * p.head_rows : 0);
        const uint32_t lanes = static_cast<uint32_t>(warp * 32) << 16, lane_base = tmem_base + lanes;
        const float sl2 = p.scale_log2;
        float m_run = -INFINITY, l_run = 0.f;  // running maximum of the raw scores (reference of the exponentials), sum
        const int row_limit = min(kvlen - 1, causal ? qi + causal_off : 0x7fffffff);  // last visible key of this row
#pragma unroll 1
        for (int g = 0; g < n; ++g) {
            const int key0 = g * kStep;
            if (!warp_wait(s_full, g & 1)) { failed = true; break; }
            tc_fence_after_sync();
            float s[kStep];
#pragma unroll
            for (int c = 0; c < kStep / 32; ++c) {
                uint32_t rr[32];
                tmem_ld_x32(lane_base + c * 32, rr);
#pragma unroll
                for (int k = 0; k < 32; ++k) s[c * 32 + k] = __uint_as_float(rr[k]);
            }
            tmem_ld_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(s_read);  // the next scores may take S's columns
            const int lim = row_limit - key0;  // last visible column of this step
            const bool masked = __any_sync(0xffffffffu, lim < kStep - 1);
            if (masked) {
#pragma unroll
                for (int k = 0; k < kStep; ++k) s[k] = (k <= lim) ? s[k] : -INFINITY;
            }
            float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
            for (int k = 4; k + 7 < kStep; k += 8) {
                mx[0] = max3_nan(mx[0], s[k], s[k + 1]);
                mx[1] = max3_nan(mx[1], s[k + 2], s[k + 3]);
                mx[2] = max3_nan(mx[2], s[k + 4], s[k + 5]);
                mx[3] = max3_nan(mx[3], s[k + 6], s[k + 7]);
            }
            mx[0] = max3_nan(mx[0], s[kStep - 4], s[kStep - 3]);
            mx[1] = max3_nan(mx[1], s[kStep - 2], s[kStep - 1]);
            const float m_tile = max3_nan(max3_nan(mx[0], mx[1], mx[1]), mx[2], mx[3]);  // NaN if a score is
            // Keep the old reference unless this step's maximum exceeds it by more than the threshold.  The comparison also fails for a
            // row without a reference yet, a NaN and a second +inf.
            bool exact = masked;  // no exponentials on the FMA pipe: there a score of -inf or NaN would count as a small one
            if (__any_sync(0xffffffffu, !((m_tile - m_run) * sl2 <= kRescaleThreshold))) {
                const bool grow = m_tile > -INFINITY && !((m_tile - m_run) * sl2 <= kRescaleThreshold);  // never by a NaN
                float alpha = 1.f;
                if (grow) {
                    // first visible keys of this row: nothing accumulated yet, nothing to rescale
                    alpha = (m_run == -INFINITY) ? 1.f : ex2((m_run - m_tile) * sl2);
                    m_run = m_tile;
                }
                exact = exact || __any_sync(0xffffffffu, m_tile != m_tile || fabsf(m_run) == INFINITY);
                l_run *= alpha;
                if (g > 0 && __any_sync(0xffffffffu, alpha != 1.f)) {
                    if (!warp_wait(pv_done, (g - 1) & 1)) { failed = true; break; }  // O holds every product, none is in flight
                    tc_fence_after_sync();
#pragma unroll 1
                    for (int c = 0; c < kD / 16; ++c) {
                        uint32_t rr[16];
                        tmem_ld_x16(lane_base + kColO + c * 16, rr);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 16; ++k) rr[k] = __float_as_uint(__uint_as_float(rr[k]) * alpha);
                        tmem_st_x16(lane_base + kColO + c * 16, rr);
                    }
                }
            }
            const float m_ref = (m_run == -INFINITY) ? 0.f : m_run;
            const float2 sl2v = make_float2(sl2, sl2), neg_m = make_float2(-m_ref * sl2, -m_ref * sl2);
            float2 lsum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
            uint32_t packed[32];
            auto exponentials = [&](auto fma_tag) {
                constexpr int kOnFma = decltype(fma_tag)::value;  // of the 32 pairs, evenly spaced
#pragma unroll
                for (int k = 0; k < 32; ++k) {
                    const float2 x = ffma2(make_float2(s[2 * k], s[2 * k + 1]), sl2v, neg_m);
                    const bool on_fma = ((k + 1) * kOnFma / 32) != (k * kOnFma / 32);
                    const float2 pr = on_fma ? ex2_fma2_fine(x) : make_float2(ex2(x.x), ex2(x.y));  // masked: 0
                    lsum[k & 1] = fadd2(lsum[k & 1], pr);
                    packed[k] = pack16<F16>(pr.x, pr.y);
                }
            };
            if (exact) exponentials(std::integral_constant<int, 0>{});
            else exponentials(std::integral_constant<int, kFmaExpPairs>{});
            if (g > 0) {  // the product of the step before has read its P
                if (!warp_wait(pv_done, (g - 1) & 1)) { failed = true; break; }
                tc_fence_after_sync();
            }
            tmem_st_x32(tmem_p + lanes, packed);
            l_run += (lsum[0].x + lsum[0].y) + (lsum[1].x + lsum[1].y);
            // V rows at and beyond lens[b] hold the caller's padding (possibly NaN, and 0 x NaN is NaN): zero them before the
            // product may start.  Rows beyond Skv were zero-filled by the copy itself.
            if (padding && key0 + kStep > kvlen && kvlen < p.Skv) {
                if (!warp_wait(&v_full[g % kStages], (g / kStages) & 1)) { failed = true; break; }
                uint4* vt = reinterpret_cast<uint4*>(sV + (g % kStages) * L::kKVBytes);
                for (int i = max(kvlen - key0, 0) * 8 + row; i < kStep * 8; i += 128) vt[i] = make_uint4(0, 0, 0, 0);
                fence_proxy_async_smem();
            }
            tmem_st_wait();
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(p_ready);
        }
        if (n == 0) {  // no visible key for any row of this tile: zeros, with plain stores
            if (live && qi < p.Sq) {
                uint16_t* orow = p.out + b * p.o_sb + (head + row_h) * p.o_sh + qi * p.o_ss;
                for (int c = 0; c < p.head_dim / 8; ++c) reinterpret_cast<uint4*>(orow)[c] = make_uint4(0, 0, 0, 0);
            }
        } else if (!failed && warp_wait(pv_done, (n - 1) & 1)) {  // the last product
            tc_fence_after_sync();
            // O / l as 16-bit values into Q's place (all scores are done), in the copies' 128-byte swizzle
            const float inv = l_run > 0.f ? 1.f / l_run : 0.f;
            uint8_t* line = sQ + row * 128;
#pragma unroll
            for (int c32 = 0; c32 < 2; ++c32) {
                uint32_t cur[32];
                tmem_ld_x32(lane_base + kColO + c32 * 32, cur);
                tmem_ld_wait();
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    uint32_t w[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        w[k] = pack16<F16>(__uint_as_float(cur[c * 8 + 2 * k]) * inv, __uint_as_float(cur[c * 8 + 2 * k + 1]) * inv);
                    *reinterpret_cast<uint4*>(line + (((c32 * 4 + c) ^ (row & 7)) << 4)) = make_uint4(w[0], w[1], w[2], w[3]);
                }
            }
            fence_proxy_async_smem();
            __syncwarp();
            if (rows == kBM) {  // powers of two, so a warp's rows are a box: no waiting for the other three
                const int r0 = warp * 32, q = q0 + r0 % p.head_rows;
                if (lane == 0 && q < p.Sq) tma_store_4d(&tmap_o, sQ + r0 * 128, 0, q, head + r0 / p.head_rows, b);
            } else {
                if (lane == 0) mbar_arrive(o_staged);
                if (warp == 0) {
                    if (!warp_wait(o_staged, 0)) failed = true;
                    else if (lane == 0) tma_store_4d(&tmap_o, sQ, 0, q0, head, b);
                }
            }
            if (lane == 0) {
                tma_store_commit();
                tma_store_wait_read<0>();  // shared memory is not given up before it has been read
            }
            __syncwarp();
        } else {
            failed = true;
        }
    }

    if (failed) {
        atomicExch(p.status, 1);
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);  // let copies and MMAs in flight land
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 4) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
        tmem_dealloc(tmem_p, kTmemColsP);
    }
}

template <bool F16>
int launch_narrow(const void* q, const void* k, const void* v, void* out, int B, int Hq, int Hkv, int Sq, int Skv,
                  int head_dim, int mask_kind, const int32_t* lens, float scale, const long long (*st)[3], cudaStream_t s) {
    using L = NarrowSmem;
    auto encode = [&](CUtensorMap* m, const void* base, int H, int S, const long long* str, int box_rows, int box_heads = 1) {
        const uint32_t box[4] = {64, (uint32_t)box_rows, (uint32_t)box_heads, 1};
        const uint64_t dims[4] = {(uint64_t)head_dim, (uint64_t)S, (uint64_t)H, (uint64_t)B};
        const uint64_t strides[3] = {(uint64_t)str[2] * 2, (uint64_t)str[1] * 2, (uint64_t)str[0] * 2};
        return encode_tmap_bf16_sw128(m, base, 4, dims, strides, box);
    };
    CUtensorMap tq, tk, tv, to;
    const HeadPack hp = choose_pack(Hq / Hkv, Sq, Skv, (mask_kind & FORGE_MASK_CAUSAL) != 0, false);
    if (!encode(&tq, q, Hq, Sq, st[0], hp.rows, hp.pack)) return FORGE_ERR_CUDA;
    if (!encode(&tk, k, Hkv, Skv, st[1], kStep)) return FORGE_ERR_CUDA;
    if (!encode(&tv, v, Hkv, Skv, st[2], kStep)) return FORGE_ERR_CUDA;
    // the output leaves in boxes of a warp's rows where all 128 are in use, else of the whole tile (the kernel asks the same)
    const int warp_rows = hp.rows < 32 ? hp.rows : 32;
    const bool own = hp.pack * hp.rows == kBM;
    if (!encode(&to, out, Hq, Sq, st[3], own ? warp_rows : hp.rows, own ? 32 / warp_rows : hp.pack)) return FORGE_ERR_CUDA;
    NarrowParams p;
    p.out = static_cast<uint16_t*>(out);
    p.o_sb = st[3][0]; p.o_sh = st[3][1]; p.o_ss = st[3][2];
    p.lens = lens;
    p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.Sq = Sq; p.Skv = Skv; p.head_dim = head_dim; p.mask_kind = mask_kind;
    p.pack = hp.pack; p.head_rows = hp.rows;
    p.scale_log2 = scale * 1.4426950408889634f;
    // scale = 0 (uniform weights): any positive multiplier whose products with the scores flush to zero
    if (!(p.scale_log2 > 0.f)) p.scale_log2 = 1.17549435e-38f;
    p.status = device_status_word();
    if (!p.status) return FORGE_ERR_CUDA;
    const auto kernel = attn_narrow_kernel<F16>;
    constexpr int kAlone = 116 * 1024, kTwo = 78 * 1024;
    FORGE_SET_SMEM_ONCE(kernel, kAlone);
    const long long tiles = (long long)B * (Hq / hp.pack) * ((Sq + hp.rows - 1) / hp.rows);
    if (tiles > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    // Launched early, beside the previous kernel's, three CTAs would share an SM that is free already while others fall idle a moment
    // later.  So a grid of up to two CTAs per SM takes shared memory for two, and one that leaves a quarter of the SMs to others for one.
    // (One each for up to all SMs keeps a second stream's grid out until the first has ended.)  Three / two / one per SM, us.  Two streams, a
    // pair of calls: 8 x 12 heads x 128 (96 tiles) 5.8 / 5.2 / 6.9, 3 x 12 x 384 (108) 8.7 / 8.5 / 9.6, 12 x 12 x 128 (144) 6.0 / 5.7 / 10.0,
    // 6 x 12 x 256 (144) 7.6 / 7.1 / 11.3; the kernel before this one took 6.7, 10.5, 7.1 and 9.0.  The same call in a chain: 8 x 12 x 128
    // 5.5 / 5.1 / 4.8, 3 x 12 x 384 9.0 / 8.0 / 7.4, 12 x 12 x 128 6.1 / 5.4 / 5.1, 6 x 12 x 256 7.9 / 7.0 / 6.0.  GPT-2-small layers, 1 x 512
    // 42.5 / 40.2 / 39.1, 2 x 256 38.3 / 37.1 / 36.5, 2 x 128 31.2 / 31.7 / 31.6; layers of 32/8 heads of 64, width 2048, 2 x 128 56.7 / 56.7 /
    // 58.6 (its CTA of 116 KB sets up only when the projection's has left), 2 x 256 79.4 / 81.1 / 81.0.
    const int sms = sm_count(), smem = 4 * tiles <= 3LL * sms ? kAlone : tiles <= 2LL * sms ? kTwo : L::kAlloc;
    FORGE_CUDA_TRY(launch_pdl(kernel, dim3((unsigned)tiles), dim3(kThreads), smem, s, tq, tk, tv, to, p));
    return finish_launch(1);
}

}  // namespace

int attn_narrow(bool f16, const void* q, const void* k, const void* v, void* out, int B, int Hq, int Hkv, int Sq, int Skv,
                int head_dim, int mask_kind, const int32_t* lens, float scale, const long long (*strides)[3], cudaStream_t s) {
    return f16 ? launch_narrow<true>(q, k, v, out, B, Hq, Hkv, Sq, Skv, head_dim, mask_kind, lens, scale, strides, s)
               : launch_narrow<false>(q, k, v, out, B, Hq, Hkv, Sq, Skv, head_dim, mask_kind, lens, scale, strides, s);
}

}  // namespace forge
