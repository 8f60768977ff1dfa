// Fused attention, 16-bit in / fp32 accumulate / 16-bit out (Eq. 8 / Eq. 9): scores, mask, online
// softmax and the product with V in one kernel; S and P never reach global memory.  The element type
// is bf16 or fp16 (a template parameter: the MMA operand format and the two conversions differ).
// Head sizes 72 .. 128, and up to 64 with an additive bias or in many short tiles (many_short_tiles(); attn_narrow.cu has the rest up to 64).
//
// One work item = two 128-row query tiles (see the item decoding below).  Every 128-key tile of S is
// computed, normalised and multiplied with V in two 64-key halves with their own barriers, so each
// query tile has two independent half-step streams and the CTA has four: while a softmax thread works
// on one half, the tensor core multiplies the other half's P with V and produces that half's next S.
// Warp roles:
//   warps 0-3 : softmax / rescale / epilogue of tile 0; thread = one query row (TMEM lane), so row
//   warps 4-7 : the same for tile 1                    maxima and sums need no cross-thread reduction
//   warp 8    : TMA producer: Q tiles, then K and V tiles (64 keys, one per half-step) through rings;
//               it sleeps between barrier polls (a spinning thread takes issue slots from the softmax
//               warp of its scheduler: 1.2 % of the kernel)
//   warp 9    : tcgen05.mma issuer of tile 0 (one elected lane), owns the TMEM allocation
//   warp 10   : tcgen05.mma issuer of tile 1
//   warp 11   : issues the TMA stores of both tiles' outputs (but the last ones); the third warpgroup hands registers to the other two
//   (setmaxnreg: 208 per softmax thread, 88 for the rest; 256*208 + 128*88 = 384*168 as launched).
// Tensor memory (512 columns): S_t at t*128 (half h at +64h, 64 fp32 columns each), O_0 at 256,
// O_1 at 256 + D.  P (bf16, two per column) of half h is written over the first 32 columns of that
// half of S and is the A operand of the P V product straight from tensor memory.  A tile's issuer
// thread issues, per half-step g (key tile g/2, half g%2):  O += P(g) V(g), then S(g+2) = Q K(g+2)^T.
// MMAs of one thread execute in issue order, so P(g) is read before S(g+2) overwrites it, and the
// barrier that announces S(g+2) also covers the completion of the P V products up to g.
// O is rescaled in TMEM only when a row's maximum grows by more than 2^8 (the stale maximum is
// kept otherwise; the final division by l uses the same reference, so the result is unchanged).
// Q and K are K-major operands, V [keys, D] is the MN-major B operand of P V.
// Between items: each tile has two Q buffers, so the issuer sends the first two scores of the next item right behind
// the last products of this one; the output is staged in the Q buffer of its own item (whose last reader was that item's
// last S) and stored from there by warp 11, which then hands the buffer back.  A boundary costs the softmax warps
// about 3100 cycles instead of 4700 (18 x 32/8 x 895 x 96 padded 153 -> 149 us).
// The CTA's last output is stored by the softmax warps, each its own rows, without the way through warp 11: with one item
// per CTA that is 0.4 us (6 x 12 heads x 385 causal, D = 128, 12.56 -> 12.15).
// Reading the output only after the next item's first half-step gained nothing more and cost short items their overlap
// (64 x 16/4 x 64: 16.7 -> 21.3 us).  At D = 128 a run of seconds is at the power limit (4 x 32/8 x 2048 130 us at 1965 MHz in a few calls,
// 150 at 1620 MHz later on): there fewer cycles are a lower clock.
#include <type_traits>

#include "attn_math.cuh"
#include "attn_narrow.cuh"
#include "attn_tiles.cuh"
#include "attn_wide.cuh"
#include "forge_common.cuh"
#include "sm100_ptx.cuh"
#include "tmap.cuh"

namespace forge {
namespace {

using namespace ptx;

constexpr int kBM = 128;          // query rows per tile
constexpr int kTilesPerCta = 2;
constexpr int kBN = 128;          // keys per tile of S (two half-steps)
constexpr int kHalf = 64;         // keys per half-step and per K/V tile in shared memory
constexpr int kThreads = 384;
constexpr int kTmemCols = 512;
constexpr int kColS = 0;          // S_t at t * 128
constexpr int kColO = 256;        // O_t at 256 + t * D
constexpr int kTakeAhead = 6;     // half-steps before the end of an item's loads at which the next item is taken
constexpr float kRescaleThreshold = 8.0f;  // log2 units
#ifndef FORGE_ATTN_FMA_EXP_PAIRS
#define FORGE_ATTN_FMA_EXP_PAIRS 2
#endif
// of the 32 score pairs of a half-step, how many take their exponentials on the FMA pipe (unmasked steps)
constexpr int kFmaExpPairs = FORGE_ATTN_FMA_EXP_PAIRS;

template <int D>
struct AttnSmem {
    static constexpr int kChunkBytes = 128 * 128;              // Q: 128 rows x 64 bf16 (one swizzle span wide)
    static constexpr int kTileBytes = (D / 64) * kChunkBytes;  // a Q tile
    static constexpr int kKVChunkBytes = kHalf * 128;          // K, V: 64 keys x 64 bf16
    static constexpr int kKVTileBytes = (D / 64) * kKVChunkBytes;
    static constexpr int kKVStages = (D == 64) ? 8 : 3;
    static constexpr int kQOff = 0;
    static constexpr int kKOff = kQOff + 2 * kTilesPerCta * kTileBytes;  // two Q buffers per tile
    static constexpr int kVOff = kKOff + kKVStages * kKVTileBytes;
    static constexpr int kBarOff = kVOff + kKVStages * kKVTileBytes;
    // q_full[4], q_empty[4], k/v full+empty per stage, s_full[4], p_ready[4], pv_done[4], o_free[2], next_full[2],
    // next_empty[2], taken, o_staged[4]
    static constexpr int kNumBars = 8 + 4 * kKVStages + 23;
    static constexpr int kNextOff = kBarOff + (kNumBars * 8 + 15) / 16 * 16;  // the launch queue's answer, two items
    static constexpr int kTotal = kNextOff + 16 + 2 * 64 + 16;
    static constexpr int kAlloc = kTotal + 1024;
};

// Division by a divisor fixed at launch: floor(n / d) = high 64 bits of n * ceil(2^64 / d) for 0 <= n < 2^32.
struct FastDiv {
    unsigned long long m;  // ceil(2^64 / d); unused for d == 1
    int d;
};
inline FastDiv make_fastdiv(int d) {
    FastDiv f;
    f.d = d;
    f.m = d > 1 ? ~0ull / (unsigned long long)d + 1ull : 0ull;
    return f;
}
__device__ __forceinline__ int fast_div(int n, const FastDiv& f) {
    return f.d == 1 ? n : (int)__umul64hi((unsigned long long)(unsigned)n, f.m);
}

struct AttnParams {
    uint16_t* out;  // bf16 or fp16 elements
    long long o_sb, o_sh, o_ss;  // element strides of out between batch entries, heads and rows
    const int32_t* lens;
    const float* bias;  // additive bias on the scaled scores [B, bias_heads, Sq, Skv], or nullptr
    const float* bias_end;  // one past its last element
    int bias_heads;     // 1 (shared by all heads) or Hq
    float inv_scale;    // 1 / scale: the bias is added to the unscaled scores as bias / scale
    int B, Hq, Hkv, Sq, Skv;
    int head_dim;  // elements per row in memory (<= the kernel's D; the TMA unit zero-fills the difference)
    int mask_kind;
    float scale_log2;  // > 0 (a zero scale is passed as the smallest normal number: every product flushes to 0)
    int pack, head_rows;  // query heads in a tile and the rows of each (attn_tiles.cuh)
    int tiles;            // query tiles of an item (1 or 2)
    int steps, inner;     // items of a head group, head groups (two_streams: head pairs) per batch entry
    FastDiv div_heads;  // by the number of items per query step
    FastDiv div_inner;  // by `inner`
    FastDiv div_group;  // by the query heads per KV head
    int sms, dynamic;   // dynamic: more items than SMs
    int* status;
};

// What one CTA needs to know about a work item (a pair of query tiles).
struct ItemInfo {
    int b, kvlen;
    int kvh[kTilesPerCta];      // KV head of each tile (equal unless the tiles read separate K/V streams)
    int q0[kTilesPerCta];       // first query row of each of the two tiles
    int h[kTilesPerCta];        // (first) query head of each tile
    int nh[kTilesPerCta];       // 64-key half-steps visible to at least one row of each query tile (0: no work)
    int n_max;                  // the larger of the two
};

// element t of a two-element array without dynamic indexing (keeps the array in registers)
__device__ __forceinline__ int pick(const int (&a)[kTilesPerCta], int t) { return t ? a[1] : a[0]; }

// PACK: several heads per tile.  (A parameter, because the instance with one head per tile is slower when it carries the divisions along:
// 6 x 12 x 385 causal, D = 128, 12.6 -> 13.0 us.)
template <int D, bool F16, bool BIAS, bool PACK>
__global__ void __launch_bounds__(kThreads, 1)
attn_bf16_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                 const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ CUtensorMap tmap_o,
                 const __grid_constant__ CUtensorMap tmap_o32, const AttnParams p) {
    using L = AttnSmem<D>;
    constexpr int kKVStages = L::kKVStages;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* sQ = smem + L::kQOff;
    uint8_t* sK = smem + L::kKOff;
    uint8_t* sV = smem + L::kVOff;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kBarOff);
    uint64_t* q_full = bars;                 // [4] query tile t, buffer u at t * 2 + u
    uint64_t* q_empty = bars + 4;            // [4] the output that was staged in the buffer has left it
    uint64_t* k_full = bars + 8;
    uint64_t* k_empty = k_full + kKVStages;
    uint64_t* v_full = k_empty + kKVStages;
    uint64_t* v_empty = v_full + kKVStages;
    uint64_t* s_full = v_empty + kKVStages;  // [4] query tile t, half h at t * 2 + h
    uint64_t* p_ready = s_full + 4;          // [4]
    uint64_t* pv_done = p_ready + 4;         // [4] one completion per P V product of that tile and half
    uint64_t* o_free = pv_done + 4;          // [2] per query tile
    uint64_t* next_full = o_free + 2;        // [2] the next item is in shared memory (two places in turn)
    uint64_t* next_empty = next_full + 2;    // [2] both issuers, the eight softmax warps and the store warp have read it
    uint64_t* taken = next_empty + 2;        // the launch queue has answered
    uint64_t* o_staged = taken + 1;          // [4] the tile's output lies in its Q buffer, ready to be stored
    uint8_t* next_answer = smem + L::kNextOff;
    // [2][16]: 1 or 0 (no item), then b, kvlen, n_max, q0[2], h[2], nh[2] as in ItemInfo
    volatile int* next_items = reinterpret_cast<int*>(smem + L::kNextOff + 16);
    uint32_t* tmem_base_slot = reinterpret_cast<uint32_t*>(smem + L::kNextOff + 16 + 2 * 64);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // A tile holds head_rows consecutive query rows of `pack` query heads that share K and V (attn_tiles.cuh).  An item is two
    // consecutive tiles of a head group, or one (choose_tiles() has the rules).  Without packing at D = 64 (where shared memory
    // has room for it) the two tiles are two heads on the same query rows instead, each with its own K/V stream through half
    // of the stage ring.
    const int head_rows = PACK ? p.head_rows : kBM, pack = PACK ? p.pack : 1;
    const bool two_streams = !PACK && kKVStages >= 8 && (!BIAS || p.tiles == 2);  // (without a bias always two tiles: choose_tiles())
    const int ring_len = two_streams ? kKVStages / 2 : kKVStages;
    const int heads = p.inner * p.B;  // items per query step
    const uint32_t q_bytes = (uint32_t)(pack * head_rows) * (D * 2);
    // ring slot and phase of the g-th KV tile of stream u
    auto kv_slot = [&](int u, int g) { return (two_streams ? u * ring_len : 0) + g % ring_len; };
    auto kv_phase = [&](int g) { return (uint32_t)((g / ring_len) & 1); };
    const int causal_off = p.Skv - p.Sq;
    const bool causal = (p.mask_kind & FORGE_MASK_CAUSAL) != 0;

    // Dynamic schedule.  The grid has one CTA per item, ordered longest first (the last query-tile pair of every head, then
    // the one before, ...); a CTA that nears the end of its item takes the next one that has not started yet out of the
    // launch queue, so whoever is done first gets it, whatever the items cost (padding, ragged tiles).  Against a fixed
    // order (item c of every round to CTA c, in alternating direction): 8 x 16/4 heads x 1000 x 1700 with lengths from 300
    // 74 -> 66 us, 2 x 28/4 x 2048 causal 65.6 -> 62.7, 8 x 12 x 1024 causal (an even load) 34.5 -> 34.1.
    // (What the softmax loop gets for registers hangs on where this comes from: without packing a flag from the host costs 3 %, 2 x 16 x
    // 4000 not causal 247 -> 254 us; with it the comparison does, 1 x 32/8 x 4096 243 -> 250.)
    const bool dynamic = PACK ? p.dynamic != 0 : p.steps * heads > p.sms;  // else everything runs at once and nothing is left to take
    auto decode = [&](int i) {
        ItemInfo it;
        const int round_q = fast_div(i, p.div_heads);
        const int qstep = p.steps - 1 - round_q;  // longest (causal) first
        const int hb = i - round_q * heads;
        it.b = fast_div(hb, p.div_inner);
        const int in_b = hb - it.b * p.inner;
        if (two_streams) {
            it.h[0] = 2 * in_b;
            it.h[1] = min(2 * in_b + 1, p.Hq - 1);
            it.q0[0] = qstep * kBM;
            it.q0[1] = 2 * in_b + 1 < p.Hq ? it.q0[0] : p.Sq;  // odd head count: no second tile
        } else {
            it.h[0] = it.h[1] = in_b * pack;
            it.q0[0] = p.tiles * qstep * head_rows;
            it.q0[1] = p.tiles == 2 ? it.q0[0] + head_rows : p.Sq;
        }
        it.kvh[0] = fast_div(it.h[0], p.div_group);
        it.kvh[1] = fast_div(it.h[1], p.div_group);
        it.kvlen = p.Skv;
        if (p.mask_kind & FORGE_MASK_PADDING) it.kvlen = min(max(p.lens[it.b], 0), p.Skv);
        it.n_max = 0;
#pragma unroll
        for (int t = 0; t < kTilesPerCta; ++t) {
            const int q0 = it.q0[t];
            int kv_end = it.kvlen;
            if (causal) kv_end = min(kv_end, min(q0 + head_rows, p.Sq) + causal_off);
            if (q0 >= p.Sq) kv_end = 0;
            kv_end = max(kv_end, 0);
            it.nh[t] = (kv_end + kHalf - 1) / kHalf;
            it.n_max = max(it.n_max, it.nh[t]);
        }
        return it;
    };
    // The n-th item after the first, worked out by the producer and read by everyone else from next_items[n % 2]: 1 if there
    // is one, 0: no more work, -1: gave up.
    auto next_item = [&](int n, bool relaxed = false) -> int {
        if (!dynamic) return 0;
        if (!(relaxed ? mbar_wait_relaxed(&next_full[n & 1], (n >> 1) & 1) : mbar_wait(&next_full[n & 1], (n >> 1) & 1))) return -1;
        return next_items[(n & 1) * 16];
    };
    // Sends the tile's rows from `row` on off, out of Q buffer `at`, where the output is staged: as many as the map's box has (all
    // rows in use, or a quarter of the tile).  Rows beyond Sq are clipped by the TMA unit.
    auto store_rows = [&](const CUtensorMap* map, int at, int row, int q, int head, int b) {
        if (q >= p.Sq) return;
#pragma unroll
        for (int c = 0; c < D / 64; ++c)
            tma_store_4d(map, sQ + at * L::kTileBytes + c * L::kChunkBytes + row * 128, c * 64, q, head, b);
        tma_store_commit();
    };

    if (threadIdx.x == 0) {
        for (int i = 0; i < 4; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); mbar_init(&o_staged[i], 4); }
        mbar_init(taken, 1);
        // a shared K/V stage is released by both tiles' issuer threads, a private one by its own
        const uint32_t releases = two_streams ? 1 : 2;
        for (int i = 0; i < kKVStages; ++i) {
            mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], releases);
            mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], releases);
        }
        for (int i = 0; i < 4; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_ready[i], 4); mbar_init(&pv_done[i], 1); }
        for (int t = 0; t < 2; ++t) { mbar_init(&o_free[t], 4); mbar_init(&next_full[t], 1); mbar_init(&next_empty[t], 11); }
        fence_mbar_init();
        prefetch_tmap(&tmap_q); prefetch_tmap(&tmap_k); prefetch_tmap(&tmap_v); prefetch_tmap(&tmap_o); prefetch_tmap(&tmap_o32);
    }
    if (warp == 9) {
        tmem_alloc(tmem_base_slot, kTmemCols);
        tmem_relinquish();
    }
    // Rows of a Q tile that are not in use are never written by the copies: zero scores, not whatever lies there.
    if constexpr (PACK) {
        for (int r = pack * head_rows + (int)threadIdx.x / 8; r < kBM; r += kThreads / 8)
            for (int c = 0; c < 2 * kTilesPerCta * (D / 64); ++c)
                *reinterpret_cast<uint4*>(sQ + c * L::kChunkBytes + r * 128 + (threadIdx.x % 8) * 16) = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem_base = *tmem_base_slot;
    bool failed = false;
    // set-up done: the next kernel may move in as SMs free up; nothing global is touched before the
    // previous kernel has completed
    pdl_launch_dependents();
    pdl_wait();

    if (warp >= 8) {
      asm volatile("setmaxnreg.dec.sync.aligned.u32 88;");
      if (warp == 8) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int kvn[2] = {0, 0};     // KV tiles loaded so far per stream (ring position), across items
            int q_loads[2] = {0, 0}; // Q tiles loaded so far per query tile
            auto load_q = [&](const ItemInfo& x) -> bool {
#pragma unroll
                for (int t = 0; t < kTilesPerCta; ++t) {
                    if (x.nh[t] == 0) continue;
                    const int u = q_loads[t] & 1, at = t * 2 + u;
                    if (!mbar_wait_relaxed(&q_empty[at], ((q_loads[t] >> 1) & 1) ^ 1)) return false;
                    ++q_loads[t];
                    mbar_expect_tx(&q_full[at], q_bytes);
#pragma unroll
                    for (int c = 0; c < D / 64; ++c)  // rows beyond Sq are zero-filled by the TMA unit
                        tma_load_4d(sQ + at * L::kTileBytes + c * L::kChunkBytes, &tmap_q, &q_full[at], c * 64, x.q0[t], x.h[t], x.b);
                }
                return true;
            };
            ItemInfo it = decode(blockIdx.x), nx = it;
            if (!load_q(it)) failed = true;
            bool more = true;
            for (int r = 0; more && !failed; ++r) {
                more = false;
                // takes the next item out of the launch queue / publishes it
                auto request_next = [&]() {
                    mbar_expect_tx(taken, 16);
                    clc_try_cancel(next_answer, taken);
                };
                auto receive_next = [&]() -> bool {
                    if (!mbar_wait(taken, r & 1)) return false;
                    const int x = clc_taken(next_answer);
                    fence_proxy_async_smem();  // the next answer is written to this place by another proxy
                    more = x >= 0;
                    if (more) nx = decode(x);
                    if (!mbar_wait_relaxed(&next_empty[r & 1], ((r >> 1) & 1) ^ 1)) return false;
                    volatile int* to = next_items + (r & 1) * 16;
                    to[0] = more ? 1 : 0; to[1] = nx.b; to[2] = nx.kvlen; to[3] = nx.n_max;
                    to[4] = nx.q0[0]; to[5] = nx.q0[1]; to[6] = nx.h[0]; to[7] = nx.h[1]; to[8] = nx.nh[0]; to[9] = nx.nh[1];
                    mbar_arrive(&next_full[r & 1]);
                    // its Q tiles are asked into L2 while their buffer may still be in use
#pragma unroll
                    for (int t = 0; t < kTilesPerCta; ++t) {
                        if (!more || nx.nh[t] == 0) continue;
#pragma unroll
                        for (int c = 0; c < D / 64; ++c) tma_prefetch_l2_4d(&tmap_q, c * 64, nx.q0[t], nx.h[t], nx.b);
                    }
                    return true;
                };
                // Late enough that the item goes to whoever is done first, early enough that its Q tiles, which are loaded behind
                // this item's last K/V tiles, are in shared memory before the last products of this one are out.  The answer
                // of the launch queue is not waited for before the first K/V tiles are on their way.
                const int j_request = max(0, it.n_max - kTakeAhead);
                const int j_receive = it.n_max > kTakeAhead / 2 ? it.n_max - kTakeAhead / 2 : it.n_max;
                if (dynamic && it.n_max == 0) request_next();
                for (int j = 0; j < it.n_max && !failed; ++j) {
                    if (dynamic && j == j_request) request_next();
                    if (dynamic && j == j_receive && !receive_next()) { failed = true; break; }
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        if (u == 1 && !two_streams) continue;
                        if (two_streams && j >= it.nh[u]) continue;
                        const int g = kvn[u]++, st = kv_slot(u, g);
                        const uint32_t ph = kv_phase(g);
                        const int kvh = it.kvh[u];
                        if (!mbar_wait_relaxed(&k_empty[st], ph ^ 1)) { failed = true; break; }
                        mbar_expect_tx(&k_full[st], L::kKVTileBytes);
#pragma unroll
                        for (int c = 0; c < D / 64; ++c)
                            tma_load_4d(sK + st * L::kKVTileBytes + c * L::kKVChunkBytes, &tmap_k, &k_full[st], c * 64,
                                        j * kHalf, kvh, it.b);
                        if (!mbar_wait_relaxed(&v_empty[st], ph ^ 1)) { failed = true; break; }
                        mbar_expect_tx(&v_full[st], L::kKVTileBytes);
#pragma unroll
                        for (int c = 0; c < D / 64; ++c)
                            tma_load_4d(sV + st * L::kKVTileBytes + c * L::kKVChunkBytes, &tmap_v, &v_full[st], c * 64,
                                        j * kHalf, kvh, it.b);
                    }
                }
                if (dynamic && !failed && j_receive == it.n_max && !receive_next()) failed = true;
                // (The buffer is free once the output that was staged in it at the start of this item has left.)
                if (!failed && more && !load_q(nx)) failed = true;
                it = nx;
            }
        }
      } else if (warp <= 10) {
        // ------------------------------------------------------------------ MMA issuer of query tile t
        if (elect_one()) {
            const int t = warp - 9;
            const int u = two_streams ? t : 0;
            constexpr uint32_t idesc_s = F16 ? make_idesc_f16(kBM, kHalf, false, false) : make_idesc_bf16(kBM, kHalf, false, false);
            constexpr uint32_t idesc_o = F16 ? make_idesc_f16(kBM, D, false, true) : make_idesc_bf16(kBM, D, false, true);
            const uint32_t q_addr = smem_u32(sQ) + 2 * t * L::kTileBytes, k_addr = smem_u32(sK), v_addr = smem_u32(sV);
            const uint32_t s_tmem = tmem_base + kColS + t * kBN, o_tmem = tmem_base + kColO + t * D;
            // descriptors differ only in the start-address field: build one per operand, then add
            // (byte offset >> 4) for each step (the field cannot overflow below 256 KB)
            const uint64_t qd0 = make_smem_desc(q_addr, 16, 1024);
            int kvbase = 0;      // ring position of the item's first KV tile in this tile's stream
            int q_uses = 0;      // items in which this tile had work (Q buffers, phases of q_full, o_free)
            int steps = 0;       // half-steps of earlier items (step s uses half s % 2 of S_t, phase s / 2)
            int primed = 0;      // scores of the current item that were issued during the previous one

            // A barrier poll costs a few hundred cycles even on a completed phase, so the operands of a step
            // (V(g) for the product, K(g + 2) for the next scores) are waited for before the probabilities,
            // while this thread has nothing to issue; once P(g) arrives the MMAs go out back to back.
            auto wait_k = [&](int pos) -> bool { return mbar_wait(&k_full[kv_slot(u, pos)], kv_phase(pos)); };
            auto wait_v = [&](int pos) -> bool { return mbar_wait(&v_full[kv_slot(u, pos)], kv_phase(pos)); };
            auto wait_q = [&](int use) -> bool { return mbar_wait(&q_full[t * 2 + (use & 1)], (use >> 1) & 1); };
            // S(step) = Q K(pos)^T into half step % 2 of S_t (Q and K have landed)
            auto issue_qk = [&](int use, int step, int pos) {
                const int hh = step & 1, st = kv_slot(u, pos);
                tc_fence_after_sync();
                const uint64_t qd = qd0 + (use & 1) * (L::kTileBytes >> 4);
                const uint64_t kd = make_smem_desc(k_addr + st * L::kKVTileBytes, 16, 1024);
#pragma unroll
                for (int kk = 0; kk < D / 16; ++kk) {
                    const uint32_t qoff = ((kk / 4) * L::kChunkBytes + (kk % 4) * 32) >> 4;
                    const uint32_t koff = ((kk / 4) * L::kKVChunkBytes + (kk % 4) * 32) >> 4;
                    mma_ss(s_tmem + hh * kHalf, qd + qoff, kd + koff, idesc_s, kk != 0);
                }
                mma_commit(&s_full[t * 2 + hh]);
                mma_commit(&k_empty[st]);                  // this tile is done with the K tile
            };
            // O_t += P(g) V(g) with P read from tensor memory (V(g) has landed)
            auto issue_pv = [&](int g) -> bool {
                const int step = steps + g, hh = step & 1, st = kv_slot(u, kvbase + g);
                if (!mbar_wait(&p_ready[t * 2 + hh], (step >> 1) & 1)) return false;
                // the first product of an item overwrites O_t: the previous item's epilogue must have read it
                if (g == 0 && !mbar_wait(&o_free[t], (q_uses & 1) ^ 1)) return false;
                tc_fence_after_sync();
                // P: 16 keys = 8 columns of packed bf16 pairs.  V: MN-major, 16 keys = two 1024-byte groups
                // (2048 bytes per step); the 64-wide chunks of D are 8 KB apart.
                const uint64_t vd = make_smem_desc(v_addr + st * L::kKVTileBytes, L::kKVChunkBytes, 1024);
                const uint32_t p_tmem = s_tmem + hh * kHalf;
                if (g == 0) mma_ts(o_tmem, p_tmem, vd, idesc_o, 0u);
                else mma_ts(o_tmem, p_tmem, vd, idesc_o, 1u);
#pragma unroll
                for (int kk = 1; kk < kHalf / 16; ++kk) mma_ts(o_tmem, p_tmem + kk * 8, vd + kk * (2048 >> 4), idesc_o, 1u);
                mma_commit(&pv_done[t * 2 + hh]);
                mma_commit(&v_empty[st]);
                return true;
            };

            int nh, n_max;
            {
                const ItemInfo it = decode(blockIdx.x);
                nh = pick(it.nh, t);
                n_max = it.n_max;
            }
            int state = 1;
            for (int r = 0; state == 1; ++r) {
                // Where this tile reads every K/V tile of the item, the first scores of the next item are issued behind the last
                // products of this one, so the softmax warps go on without a gap.  (Otherwise the tiles that only the
                // other query tile reads have to be released first, or the ring would not reach the next item.)
                const bool look_ahead = nh > 0 && (two_streams || nh == n_max);
                const int next_base = kvbase + (two_streams ? nh : n_max);
                int have_next = 0, ahead = 0, next_nh = 0;
                for (int g = primed; g < min(nh, 2); ++g) {
                    if ((g == 0 && !wait_q(q_uses)) || !wait_k(kvbase + g)) { state = -1; break; }
                    issue_qk(q_uses, steps + g, kvbase + g);
                }
                for (int g = 0; g < nh && state == 1; ++g) {
                    if (!wait_v(kvbase + g) || (g + 2 < nh && !wait_k(kvbase + g + 2)) || !issue_pv(g)) { state = -1; break; }
                    if (g + 2 < nh) {
                        issue_qk(q_uses, steps + g + 2, kvbase + g + 2);
                    } else if (look_ahead) {
                        // only what is there already: the products still to come must not wait for the next item
                        if (!have_next && dynamic && mbar_test(&next_full[r & 1], (r >> 1) & 1)) {
                            have_next = 1;
                            next_nh = next_items[(r & 1) * 16] ? next_items[(r & 1) * 16 + 8 + t] : 0;
                        }
                        const int pos = next_base + ahead, use = q_uses + 1;
                        if (ahead < next_nh && mbar_test(&q_full[t * 2 + (use & 1)], (use >> 1) & 1) &&
                            mbar_test(&k_full[kv_slot(u, pos)], kv_phase(pos))) {
                            issue_qk(use, steps + nh + ahead, pos);
                            ++ahead;
                        }
                    }
                }
                if (state == -1) break;
                if (!two_streams) {
                    // K/V tiles that only the other query tile reads: release them once they have landed
                    for (int j = nh; j < n_max; ++j) {
                        const int pos = kvbase + j, st = kv_slot(0, pos);
                        if (!wait_k(pos)) { state = -1; break; }
                        mbar_arrive(&k_empty[st]);
                        if (!wait_v(pos)) { state = -1; break; }
                        mbar_arrive(&v_empty[st]);
                    }
                    if (state == -1) break;
                }
                if (nh > 0) ++q_uses;
                steps += nh;
                kvbase = next_base;
                primed = ahead;
                state = next_item(r);
                if (state == 1) {
                    nh = next_items[(r & 1) * 16 + 8 + t];
                    n_max = next_items[(r & 1) * 16 + 3];
                    mbar_arrive(&next_empty[r & 1]);
                }
            }
            if (state == -1) failed = true;
        }
      } else {
        // ------------------------------------------------------------------ output stores
        if (elect_one()) {
            int uses[2] = {0, 0};  // items in which the tile had work
            int nh[2], q0[2], h[2], b;
            {
                const ItemInfo it = decode(blockIdx.x);
                nh[0] = it.nh[0]; nh[1] = it.nh[1]; q0[0] = it.q0[0]; q0[1] = it.q0[1]; h[0] = it.h[0]; h[1] = it.h[1]; b = it.b;
            }
            for (int r = 0;; ++r) {
                int state = next_item(r, /*relaxed=*/true);
                if (state == 1) {
#pragma unroll
                    for (int t = 0; t < kTilesPerCta; ++t) {
                        if (nh[t] == 0 || state != 1) continue;
                        // (one barrier per buffer: the output of an item may be ready before the one before it has been looked at)
                        const int at = t * 2 + (uses[t] & 1);
                        if (!mbar_wait_relaxed(&o_staged[at], (uses[t] >> 1) & 1)) { state = -1; continue; }
                        ++uses[t];
                        store_rows(&tmap_o, at, 0, q0[t], h[t], b);
                        tma_store_wait_read<0>();
                        mbar_arrive(&q_empty[at]);  // the producer may load Q there again
                    }
                }
                if (state == -1) failed = true;
                if (state != 1) break;  // (the output of the last item is stored by the softmax warps)
                volatile const int* x = next_items + (r & 1) * 16;
                b = x[1]; q0[0] = x[4]; q0[1] = x[5]; h[0] = x[6]; h[1] = x[7]; nh[0] = x[8]; nh[1] = x[9];
                mbar_arrive(&next_empty[r & 1]);
            }
            tma_store_wait_all<0>();  // every output tile has left shared memory and is written
        }
      }
    } else {
        // ------------------------------------------------------------------ softmax / rescale / epilogue
        asm volatile("setmaxnreg.inc.sync.aligned.u32 208;");
        const int t = warp >> 2;       // query tile of this warp group
        const int quarter = warp & 3;  // TMEM lane quarter this warp may access
        const int row = quarter * 32 + lane;
        // this thread's query row and head within the tile; a row that is not in use goes along as the last head's row 0 with Q = 0
        // (one word: row, head * 256, in use * 65536)
        const int row_at = row < pack * head_rows ? row % head_rows + row / head_rows * 256 + 65536 : (pack - 1) * 256;
        auto row_q = [&]() { return PACK ? row_at & 255 : row; };
        auto row_h = [&]() { return PACK ? (row_at >> 8) & 255 : 0; };
        auto live = [&]() { return PACK ? row_at >= 65536 : true; };
        const uint32_t lane_base = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t col_s = kColS + t * kBN, col_o = kColO + t * D;
        const float sl2 = p.scale_log2;
        const float2 sl2v = make_float2(sl2, sl2);
        int steps = 0;               // half-steps of earlier items (step s uses half s % 2 of S_t, phase s / 2)
        int q_uses = 0;              // earlier items in which this tile had work: they use the two Q buffers in turn
        const int u = two_streams ? t : 0;  // K/V stream of this tile
        int kvbase = 0;              // ring position of the item's first KV tile in that stream
        const bool padding = (p.mask_kind & FORGE_MASK_PADDING) != 0;
        // The output of an item is read from tensor memory at the start of the next one (or of a last, empty pass): by then its
        // last products are done, and the next item's first scores have been issued behind them.
        bool pending = false;
        float out_inv = 0.f;

        int nh, q0, head, b, kvlen, n_max;
        {
            const ItemInfo it = decode(blockIdx.x);
            nh = pick(it.nh, t); q0 = pick(it.q0, t); head = pick(it.h, t);
            b = it.b; kvlen = it.kvlen; n_max = it.n_max;
        }
        for (int r = 0, state = 1; !failed; ++r) {
            const int qi = q0 + row_q();
            float m_run = -INFINITY;  // running maximum of the raw scores (reference of the exponentials)
            float l_run = 0.f;
            // last visible key of this row
            const int row_limit = min(kvlen - 1, causal ? qi + causal_off : 0x7fffffff);
            if (pending) {
                // The last product of that item (its barrier's phase before it was covered by the last S barrier seen).
                if (!warp_wait(&pv_done[t * 2 + ((steps - 1) & 1)], ((steps - 1) >> 1) & 1)) { failed = true; break; }
                tc_fence_after_sync();
                // O / l as bf16 through 128-byte-swizzled staging rows (32 rows x 64 columns per block of D) in the item's own Q
                // buffer, whose last reader was the item's last S.  A short rolled loop: its footprint matters more than its issue count.
                uint8_t* stage_out = sQ + (t * 2 + ((q_uses - 1) & 1)) * L::kTileBytes + quarter * 4096;
                uint32_t cur[32];
                tmem_ld_x32(lane_base + col_o, cur);
#pragma unroll 1
                for (int c32 = 0; c32 < D / 32; ++c32) {
                    tmem_ld_wait();
                    uint32_t w[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        w[k] = pack16<F16>(__uint_as_float(cur[2 * k]) * out_inv, __uint_as_float(cur[2 * k + 1]) * out_inv);
                    if (c32 + 1 < D / 32) tmem_ld_x32(lane_base + col_o + (c32 + 1) * 32, cur);
                    // 32 columns = four 16-byte chunks of this row's 128-byte line in block c32 / 2
                    uint8_t* line = stage_out + (c32 >> 1) * L::kChunkBytes + lane * 128;
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        *reinterpret_cast<uint4*>(line + ((((c32 & 1) * 4 + c) ^ (lane & 7)) << 4)) =
                            make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
                }
                // O_t is in shared memory: the issuer may overwrite it, the store warp may send it off
                tc_fence_before_sync();
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) { mbar_arrive(&o_free[t]); mbar_arrive(&o_staged[t * 2 + ((q_uses - 1) & 1)]); }
            }
            if (state != 1) {  // the CTA's last item (q0, head and b are still its own)
                if (pending) {
                    const int at = t * 2 + ((q_uses - 1) & 1), r0 = quarter * 32;
                    if (pack * head_rows == kBM) {  // powers of two, so a warp's rows are a box: no waiting for the other three
                        if (lane == 0) store_rows(&tmap_o32, at, r0, q0 + r0 % head_rows, head + r0 / head_rows, b);
                    } else if (quarter == 0) {
                        if (!warp_wait(&o_staged[at], ((q_uses - 1) >> 1) & 1)) { failed = true; break; }
                        if (lane == 0) store_rows(&tmap_o, at, 0, q0, head, b);
                    }
                    if (lane == 0) tma_store_wait_all<0>();  // shared memory is not given up before it has been read
                }
                break;
            }
            pending = false;
            // One half-step.  At D = 64 the first one of an item has code of its own, without the votes and branches that its
            // state decides (64 x 16 heads x 128 causal, with a fixed choice of two_streams, 18.3 -> 18.0 us; 64 x 12 x 192 25.6 -> 24.6); at
            // D = 128 and with a bias the second copy of the code costs as much as it saves.
            constexpr bool kOwnFirst = D == 64 && !BIAS;
            auto do_step = [&](auto first_tag, int g) -> bool {
                constexpr bool kFirst = decltype(first_tag)::value;
                const int step = steps + g, hh = step & 1;
                const uint32_t col_h = col_s + hh * kHalf;
                const int key0 = g * kHalf;
                // The bias of this row and half-step is on its way while the scores are waited for (4 x 16 heads x 700 x 900, a
                // bias per head: 68.9 -> 48.4 us).  Always in pieces of 16 bytes: where rows start between two of them, from the
                // piece that holds the row's first element on, and the elements are moved up below.  (One by one, each 32-byte sector
                // is asked for eight times, and the L1 left beside 224 KB of shared memory does not hold what eight warps ask for:
                // 4 x 32/8 heads x 3283, D = 96, 2243 -> 889 us; 2317 x 2321, 28/4 heads, D = 64, 163 -> 111.)
                [[maybe_unused]] float bias[BIAS ? kHalf + 4 : 1];
                [[maybe_unused]] int lead = 0;  // elements of the first piece that lie before the row's first
                if constexpr (BIAS) {
                    const int hb = p.bias_heads == 1 ? 0 : head + row_h();
                    const float* brow = p.bias + (((size_t)b * p.bias_heads + hb) * p.Sq + min(qi, p.Sq - 1)) * (size_t)p.Skv + key0;
                    lead = (int)(reinterpret_cast<uintptr_t>(brow) >> 2) & 3;
                    const int nvalid = lead + min(kHalf, p.Skv - key0);  // columns beyond Skv are masked below
                    if (__all_sync(0xffffffffu, brow - lead + ((nvalid + 3) & ~3) <= p.bias_end)) {
                        const float4* pieces = reinterpret_cast<const float4*>(brow - lead);
#pragma unroll
                        for (int c = 0; c <= kHalf / 4; ++c) {
                            const float4 bv = c * 4 < nvalid ? __ldg(pieces + c) : make_float4(0.f, 0.f, 0.f, 0.f);
                            bias[4 * c] = bv.x; bias[4 * c + 1] = bv.y; bias[4 * c + 2] = bv.z; bias[4 * c + 3] = bv.w;
                        }
                    } else {  // the last piece of some row would reach beyond the tensor's end
#pragma unroll
                        for (int k = 0; k < kHalf + 4; ++k) bias[k] = k >= lead && k < nvalid ? __ldg(brow - lead + k) : 0.f;
                    }
                }
                // S(g) is complete, and so is every MMA this tile's issuer issued before it: O_t holds the
                // P V products up to g - 2 and P(g - 2) has been consumed.
                if (!warp_wait(&s_full[t * 2 + hh], (step >> 1) & 1)) return false;
                tc_fence_after_sync();
                float s[kHalf];
#pragma unroll
                for (int c = 0; c < kHalf / 32; ++c) {
                    uint32_t rr[32];
                    tmem_ld_x32(lane_base + col_h + c * 32, rr);
#pragma unroll
                    for (int k = 0; k < 32; ++k) s[c * 32 + k] = __uint_as_float(rr[k]);
                }
                tmem_ld_wait();

                const bool need_mask = (key0 + kHalf > kvlen) || (causal && (key0 + kHalf - 1 > q0 + causal_off));
                if constexpr (BIAS) {
                    // Eq. 8's mask node as a tensor: scale * s + bias = scale * (s + bias / scale)
                    if ((p.Skv & 3) != 0) {
#pragma unroll
                        for (int k = 0; k < kHalf + 2; ++k) bias[k] = lead & 1 ? bias[k + 1] : bias[k];
#pragma unroll
                        for (int k = 0; k < kHalf; ++k) bias[k] = lead & 2 ? bias[k + 2] : bias[k];
                    }
#pragma unroll
                    for (int k = 0; k < kHalf; ++k) s[k] = fmaf(bias[k], p.inv_scale, s[k]);
                }
                bool stored = false;
                if (need_mask) {
                    const int lim = row_limit - key0;  // last visible column of this half
                    if (__all_sync(0xffffffffu, lim < 0)) {
                        // nothing visible for any row of this warp: P = 0
                        uint32_t zeros[32];
#pragma unroll
                        for (int k = 0; k < 32; ++k) zeros[k] = 0u;
                        tmem_st_x32(lane_base + col_h, zeros);
                        stored = true;
                    } else {
                        // a masked score of -inf gives a probability of exactly 0 below (the scale is > 0)
#pragma unroll
                        for (int k = 0; k < kHalf; ++k) s[k] = (k <= lim) ? s[k] : -INFINITY;
                    }
                }
                // Fast path (once every row of the warp has a finite reference): exponentials against the
                // current reference in the same pass that finds the maximum.  Valid as long as no row's
                // maximum exceeds its reference by more than the threshold, which is what the lazy rescale
                // tolerates anyway, and no score is NaN (nor +inf against a reference of +inf), which the exponentials on the FMA
                // pipe would drop; otherwise the half is redone below, with a new reference where one is due.
                if (!kFirst && !stored && __all_sync(0xffffffffu, m_run != -INFINITY)) {
                    auto fast_path = [&](auto fma_tag) {
                        constexpr bool kUseFma = decltype(fma_tag)::value;
                        const float2 neg_m = make_float2(-m_run * sl2, -m_run * sl2);
                        float2 lsum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                        float mx[4] = {s[0], s[1], s[2], s[3]};
                        uint32_t packed[32];
#pragma unroll
                        for (int k = 0; k < 32; ++k) {
                            const float s0 = s[2 * k], s1 = s[2 * k + 1];
                            mx[k & 3] = max3_nan(mx[k & 3], s0, s1);
                            const float2 x = ffma2(make_float2(s0, s1), sl2v, neg_m);
                            // evenly spaced pairs go to the FMA pipe, the rest to the special-function unit
                            const bool on_fma = kUseFma && ((k + 1) * kFmaExpPairs / 32) != (k * kFmaExpPairs / 32);
                            const float2 pr = !on_fma ? make_float2(ex2(x.x), ex2(x.y)) : D == 64 ? ex2_fma2_fine(x) : ex2_fma2(x);
                            lsum[k & 1] = fadd2(lsum[k & 1], pr);
                            packed[k] = pack16<F16>(pr.x, pr.y);
                        }
                        const float m_tile = max3_nan(max3_nan(mx[0], mx[1], mx[1]), mx[2], mx[3]);  // NaN if a score is
                        if (!__any_sync(0xffffffffu, !((m_tile - m_run) * sl2 <= kRescaleThreshold))) {
                            tmem_st_x32(lane_base + col_h, packed);
                            l_run += (lsum[0].x + lsum[0].y) + (lsum[1].x + lsum[1].y);
                            stored = true;
                        }
                    };
                    if (BIAS || need_mask) fast_path(std::false_type{});  // (a bias may hold -inf too)
                    else fast_path(std::true_type{});
                }
                if (!stored) {
                    // row maximum: four independent chains of 3-input maxima
                    float mx[4] = {s[0], s[1], s[2], s[3]};
#pragma unroll
                    for (int k = 4; k + 7 < kHalf; k += 8) {
                        mx[0] = max3(mx[0], s[k], s[k + 1]);
                        mx[1] = max3(mx[1], s[k + 2], s[k + 3]);
                        mx[2] = max3(mx[2], s[k + 4], s[k + 5]);
                        mx[3] = max3(mx[3], s[k + 6], s[k + 7]);
                    }
                    mx[0] = max3(mx[0], s[kHalf - 4], s[kHalf - 3]);
                    mx[1] = max3(mx[1], s[kHalf - 2], s[kHalf - 1]);
                    const float m_tile = max3(fmaxf(mx[0], mx[1]), mx[2], mx[3]);

                    // Keep the old reference unless this half's maximum exceeds it by more than the
                    // threshold (in log2 units of the scaled scores); then every later exponent is <= 8.
                    float alpha = 1.f;
                    bool grow = (m_tile - m_run) * sl2 > kRescaleThreshold || m_run == -INFINITY;
                    if (m_tile == -INFINITY) grow = false;
                    if (grow) {
                        // first visible keys of this row: nothing accumulated yet, nothing to rescale
                        alpha = (m_run == -INFINITY) ? 1.f : ex2((m_run - m_tile) * sl2);
                        m_run = m_tile;
                    }
                    if (!kFirst && (kOwnFirst || g > 0) && __any_sync(0xffffffffu, alpha != 1.f)) {
                        // O_t must hold every product issued so far and none may be in flight: the product of
                        // half-step g - 1 (the other half's latest) is the only one the barrier above does not cover.
                        if (!warp_wait(&pv_done[t * 2 + (hh ^ 1)], ((step - 1) >> 1) & 1)) return false;
                        tc_fence_after_sync();
                        // rare after the first steps: small chunks, not unrolled, to keep register pressure low
#pragma unroll 1
                        for (int c = 0; c < D / 16; ++c) {
                            uint32_t rr[16];
                            tmem_ld_x16(lane_base + col_o + c * 16, rr);
                            tmem_ld_wait();
#pragma unroll
                            for (int k = 0; k < 16; ++k) rr[k] = __float_as_uint(__uint_as_float(rr[k]) * alpha);
                            tmem_st_x16(lane_base + col_o + c * 16, rr);
                        }
                    }
                    const float m_ref = (m_run == -INFINITY) ? 0.f : m_run;
                    const float2 neg_m = make_float2(-m_ref * sl2, -m_ref * sl2);
                    float2 lsum[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    // P = 2^(s * sl2 - m * sl2) as packed bf16 pairs, written over the first 32 columns of this
                    // half of S_t
                    uint32_t packed[32];
#pragma unroll
                    for (int k = 0; k < 32; ++k) {
                        const float2 x = ffma2(make_float2(s[2 * k], s[2 * k + 1]), sl2v, neg_m);
                        const float2 pr = make_float2(ex2(x.x), ex2(x.y));
                        lsum[k & 1] = fadd2(lsum[k & 1], pr);
                        packed[k] = pack16<F16>(pr.x, pr.y);
                    }
                    tmem_st_x32(lane_base + col_h, packed);
                    const float l_tile = (lsum[0].x + lsum[0].y) + (lsum[1].x + lsum[1].y);
                    l_run = l_run * alpha + l_tile;
                }
                // Rows of the V tile at and beyond lens[b] were copied from the caller's padding, which may hold
                // anything; their probabilities are exactly 0, but 0 x NaN is NaN on the tensor core.  The four
                // warps of the tile zero those rows in shared memory before the product is allowed to start (the
                // issuer needs all four arrivals below).  Rows beyond Skv were zero-filled by the copy itself.
                if (padding && key0 + kHalf > kvlen && kvlen < p.Skv) {
                    const int pos = kvbase + g, st = kv_slot(u, pos);
                    if (!warp_wait(&v_full[st], kv_phase(pos))) return false;
                    const int first = max(kvlen - key0, 0);       // first padded row of this tile
                    const int per_chunk = (kHalf - first) * 8;        // 16-byte pieces to clear per 64-column chunk
                    uint8_t* vt = sV + st * L::kKVTileBytes;
                    for (int i = quarter * 32 + lane; i < (D / 64) * per_chunk; i += 128) {
                        const int c = i / per_chunk, rem = i - c * per_chunk;
                        *reinterpret_cast<uint4*>(vt + c * L::kKVChunkBytes + (first + (rem >> 3)) * 128 + ((rem & 7) << 4)) =
                            make_uint4(0, 0, 0, 0);
                    }
                    fence_proxy_async_smem();  // the tensor core reads what these threads wrote
                }
                tmem_st_wait();
                tc_fence_before_sync();
                __syncwarp();
                if (lane == 0) mbar_arrive(&p_ready[t * 2 + hh]);  // one arrival per warp
                return true;
            };
            int g = 0;
            if constexpr (kOwnFirst) {
                if (nh > 0 && !do_step(std::true_type{}, 0)) { failed = true; break; }
                g = 1;
            }
#pragma unroll 1
            for (; g < nh; ++g)
                if (!do_step(std::false_type{}, g)) { failed = true; break; }
            if (failed) break;
            if (nh > 0) {
                pending = true;
                out_inv = l_run > 0.f && live() ? 1.f / l_run : 0.f;  // no visible key, row not in use (its Q stays 0): zeros
                ++q_uses;
                steps += nh;
            } else if (live() && qi < p.Sq) {  // no visible key for any row of this tile
                uint16_t* orow = p.out + b * p.o_sb + (head + row_h()) * p.o_sh + qi * p.o_ss;
                for (int c = 0; c < p.head_dim / 8; ++c) reinterpret_cast<uint4*>(orow)[c] = make_uint4(0, 0, 0, 0);
            }
            kvbase += two_streams ? nh : n_max;
            state = next_item(r);
            if (__any_sync(0xffffffffu, state < 0)) { failed = true; break; }  // the same for every lane of the warp
            nh = 0;                // after the last item: one more pass, for its output
            if (state == 1) {
                volatile const int* x = next_items + (r & 1) * 16;
                b = x[1]; kvlen = x[2]; n_max = x[3]; q0 = x[4 + t]; head = x[6 + t]; nh = x[8 + t];
                __syncwarp();
                if (lane == 0) mbar_arrive(&next_empty[r & 1]);
            }
        }
    }

    if (failed) {
        atomicExch(p.status, 1);
        for (int i = 0; i < 2000; ++i) __nanosleep(1000);  // let copies and MMAs in flight land
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 9) {
        tc_fence_after_sync();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// Element strides of a [B, H, S, D] tensor between batch entries, heads and rows (the D elements of a row are
// contiguous).  Dense tensors have {H * S * D, S * D, D}; the strided entry point passes the caller's.
struct Strides {
    long long b, h, s;
};
inline Strides dense_strides(int H, int S, int D) { return {(long long)H * S * D, (long long)S * D, (long long)D}; }

// How the query rows are cut into tiles and items.
struct TilePlan {
    int pack, head_rows;
    bool two_streams;
    int tiles, steps, inner;
    long long items;
};

// When the last item ends, in half-steps of a pair of tiles, if at most a few short items have to wait for an SM; 0 where more do.  A lone
// tile takes 0.6 of a pair (so do the half-steps that only the later tile of an item has), an item's start and end as long as one.
inline double end_of_one_round(int pack, int B, int Hq, int Sq, int Skv, bool causal, int sms) {
    const int rows = 128 / pack, q_tiles = (Sq + rows - 1) / rows, off = Skv - Sq;
    const long long groups = (long long)(Hq / pack) * B;
    auto n = [&](int t) {  // half-steps of tile t
        const long long last = (long long)(t + 1) * rows < Sq ? (t + 1) * rows : Sq, keys = causal && last + off < Skv ? last + off : Skv;
        return keys > 0 ? (double)((keys + 63) / 64) : 0.;
    };
    auto pair = [&](int t) { return 0.6 * n(t) + 0.4 * n(t - 1); };  // tiles t and t - 1
    if (groups * q_tiles <= sms) return 0.6 * n(q_tiles - 1) + 1;
    const bool odd = q_tiles % 2 != 0;
    double longest = odd ? 0.6 * n(q_tiles - 1) : pair(q_tiles - 1);
    if (odd && q_tiles > 1 && pair(q_tiles - 2) > longest) longest = pair(q_tiles - 2);
    const long long waiting = groups * ((q_tiles + 1) / 2) - sms;
    if (waiting <= 0) return longest + 1;
    // the shortest items of all heads: those that wait start when those that do not have ended, or else the next longer ones
    if (!causal || q_tiles < 5 || waiting > groups) return 0;
    const double after = (2 * waiting <= groups ? pair(1) : pair(3)) + pair(1) + 2;
    return after > longest + 1 ? after : longest + 1;
}

// One tile per item where that leaves no SM with two of them (a lone tile takes a little more than half the time of a pair: 1 x
// 16 heads x 518 x 80 12.0 -> 10.5 us, 1 x 32/8 x 256 behind 1000 keys 25.0 -> 20.0), else two.
// choose_pack() counts scores, which is what many items cost.  Where all run at once the longest one decides, and heads that share a tile
// do not shorten it: two tiles of 128 rows start 128 keys apart, two of 18 rows see the same, and a tile of several heads takes 4 to 5 %
// longer.  us, grouped and one head per tile: 2 x 12/4 x 1100 causal 22.1 and 19.7, 1 x 28/4 x 1355 26.7 and 23.6, 2 x 28/4 x 500 13.4 and
// 12.1, 1 x 32/8 x 512 10.6 and 10.3, 2 x 16/4 x 22 4.95 and 4.49; but with few items left or one tile per item only when grouped
// 3 x 28/4 x 283 10.1 and 12.7, 2 x 10/2 x 900 15.8 and 18.0; and with a bias, which a CTA's items read once more, 2 x 16/4 x 599 53.6 and 61.3.
template <int D, bool BIAS>
TilePlan choose_tiles(int B, int Hq, int Hkv, int Sq, int Skv, int mask_kind, int sms) {
    TilePlan t;
    const bool causal = (mask_kind & FORGE_MASK_CAUSAL) != 0;
    HeadPack hp = choose_pack(Hq / Hkv, Sq, Skv, causal, true);
    if (D > 64 && !BIAS && hp.pack > 1) {
        const double one_head = end_of_one_round(1, B, Hq, Sq, Skv, causal, sms), grouped = end_of_one_round(hp.pack, B, Hq, Sq, Skv, causal, sms);
        // No diagonal whose scores grouping would save, no lone tile, and hardly fewer tiles: one head is 1 to 3 % faster (9 x 28/4 x 1737 padded,
        // D = 80, 14 tiles a head or 97 of seven, 214.8 and 209.1 us; 8 x 28/4 x 1737 of 128 233.6 and 228.6).
        const int t1 = (Sq + kBM - 1) / kBM, tp = (Sq + hp.rows - 1) / hp.rows;
        const bool level = !causal && t1 % 2 == 0 && tp > 0.98 * hp.pack * t1;
        if (level || (one_head > 0 && (grouped == 0 || one_head <= 1.07 * grouped))) hp = {1, kBM};
    }
    t.pack = hp.pack; t.head_rows = hp.rows;
    const int q_tiles = (Sq + t.head_rows - 1) / t.head_rows;
    const long long groups = (long long)(Hq / t.pack) * B;
    t.tiles = (D > 64 || BIAS) && groups * q_tiles <= sms ? 1 : 2;  // (D = 64 without a bias: always many, see many_short_tiles())
    t.two_streams = t.pack == 1 && t.tiles == 2 && AttnSmem<D>::kKVStages >= 8;  // the kernel asks the same
    t.inner = t.two_streams ? (Hq + 1) / 2 : Hq / t.pack;
    t.steps = t.two_streams ? q_tiles : (q_tiles + t.tiles - 1) / t.tiles;
    t.items = (long long)t.inner * B * t.steps;
    return t;
}

// D: the kernel's head dimension (64 or 128); head_dim <= D: the tensors' (a multiple of 8).  Columns beyond
// head_dim are zero-filled on load and clipped on store by the TMA unit, so a padded head costs time, not memory.
template <int D, bool F16, bool BIAS = false>
int launch_attn(const void* q, const void* k, const void* v, void* out, int B, int Hq, int Hkv, int Sq, int Skv,
                int head_dim, int mask_kind, const int32_t* lens, float scale, cudaStream_t s, const Strides* strides = nullptr,
                const float* bias = nullptr, int bias_heads = 1) {
    using L = AttnSmem<D>;
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    const TilePlan plan = choose_tiles<D, BIAS>(B, Hq, Hkv, Sq, Skv, mask_kind, sms);
    const Strides a = dense_strides(Hq, Sq, head_dim), c = dense_strides(Hkv, Skv, head_dim);
    const Strides sq = strides ? strides[0] : a, sk = strides ? strides[1] : c, sv = strides ? strides[2] : c, so = strides ? strides[3] : a;
    // every tensor as a 4-D map (D, rows, heads, batch): the strides carry the layout
    auto encode = [&](CUtensorMap* m, const void* base, int H, int S, const Strides& st, int box_rows, int box_heads = 1) {
        const uint32_t box[4] = {64, (uint32_t)box_rows, (uint32_t)box_heads, 1};
        const uint64_t dims[4] = {(uint64_t)head_dim, (uint64_t)S, (uint64_t)H, (uint64_t)B};
        const uint64_t strides[3] = {(uint64_t)st.s * 2, (uint64_t)st.h * 2, (uint64_t)st.b * 2};
        return encode_tmap_bf16_sw128(m, base, 4, dims, strides, box);
    };
    CUtensorMap tq, tk, tv, to, to32;
    if (!encode(&tq, q, Hq, Sq, sq, plan.head_rows, plan.pack)) return FORGE_ERR_CUDA;
    if (!encode(&tk, k, Hkv, Skv, sk, kHalf)) return FORGE_ERR_CUDA;
    if (!encode(&tv, v, Hkv, Skv, sv, kHalf)) return FORGE_ERR_CUDA;
    if (!encode(&to, out, Hq, Sq, so, plan.head_rows, plan.pack)) return FORGE_ERR_CUDA;
    const int warp_rows = plan.head_rows < 32 ? plan.head_rows : 32;  // a softmax warp's rows, where all 128 are in use
    if (!encode(&to32, out, Hq, Sq, so, warp_rows, 32 / warp_rows)) return FORGE_ERR_CUDA;
    AttnParams p;
    p.out = static_cast<uint16_t*>(out);
    p.o_sb = so.b; p.o_sh = so.h; p.o_ss = so.s;
    p.lens = lens;
    p.bias = bias;
    p.bias_end = bias ? bias + (size_t)B * bias_heads * Sq * Skv : nullptr;
    p.bias_heads = bias_heads;
    p.inv_scale = scale > 0.f ? 1.f / scale : 0.f;
    p.head_dim = head_dim;
    p.B = B; p.Hq = Hq; p.Hkv = Hkv; p.Sq = Sq; p.Skv = Skv;
    p.mask_kind = mask_kind;
    p.scale_log2 = scale * 1.4426950408889634f;
    // scale = 0 (uniform weights): any positive multiplier whose products with the scores flush to zero
    if (!(p.scale_log2 > 0.f)) p.scale_log2 = 1.17549435e-38f;
    p.status = device_status_word();
    if (!p.status) return FORGE_ERR_CUDA;
    p.pack = plan.pack; p.head_rows = plan.head_rows;
    p.tiles = plan.tiles;
    p.steps = plan.steps; p.inner = plan.inner;
    p.div_heads = make_fastdiv(plan.inner * B);
    p.div_inner = make_fastdiv(plan.inner);
    p.div_group = make_fastdiv(Hq / Hkv);
    p.sms = sms;
    p.dynamic = plan.items > sms;
    const auto packed = attn_bf16_kernel<D, F16, BIAS, true>, plain = attn_bf16_kernel<D, F16, BIAS, false>;
    const auto kernel = plan.pack > 1 ? packed : plain;
    if (plan.pack > 1) FORGE_SET_SMEM_ONCE(packed, L::kAlloc);
    else FORGE_SET_SMEM_ONCE(plain, L::kAlloc);
    FORGE_CUDA_TRY(launch_pdl(kernel, dim3((unsigned)plan.items), dim3(kThreads), L::kAlloc, s, tq, tk, tv, to, to32, p));
    return finish_launch(1);
}

// Head sizes up to 64 without a bias.  attn_narrow.cu sets up a CTA for every tile, three per SM: the better way where they all run at once
// or a tile has steps enough to hide its set-up.  Many short tiles run on this file's kernel, whose CTAs stay and fetch the next item's
// Q, K and V beside the current one's steps.  Measured, narrow and this one, us: 64 x 16 heads x 64 causal 18.4 and 14.6, x 192 35.4 and
// 29.9, x 512 (320 keys a tile) 113 and 107, x 384 not causal 85.0 and 85.0; 64 x 32/8 x 128 causal 31.3 and 23.9, padded 31.7 and 27.4.
// The other way round: 20 x 12 x 384 causal (4.9 tiles per SM; a third round of few long items) 18.2 and 20.0, x 512 (6.5) 26.3 and 26.9;
// 40 x 15 x 100 (4.1: a third round, nearly empty) 12.1 and 13.1; with a lone tile in every sixth item 26 x 16/4 x 321 22.8 and 24.5, in
// every second one 64 x 16/4 x 96 padded 13.3 and 15.6; with lengths half of the keys or less 36 x 12 x 444 38.0 and 38.6.
inline bool many_short_tiles(int B, int Hq, int Hkv, int Sq, int Skv, int mask_kind, int sms) {
    if ((long long)B * Hq * ((Sq + kBM - 1) / kBM) <= 3LL * sms) return false;  // whatever the packing (a small call's host time counts)
    const bool causal = (mask_kind & FORGE_MASK_CAUSAL) != 0, padded = (mask_kind & FORGE_MASK_PADDING) != 0;
    const HeadPack hp = choose_pack(Hq / Hkv, Sq, Skv, causal, true);
    const int q_tiles = (Sq + hp.rows - 1) / hp.rows;
    const long long tiles = (long long)B * (Hq / hp.pack) * q_tiles;
    if (tiles <= 3LL * sms || (tiles > 4LL * sms && tiles <= 5LL * sms)) return false;
    const bool lone = hp.pack > 1 && q_tiles % 2;  // the last item of a head group has one tile
    if (lone && (padded || q_tiles <= 3 || tiles <= 9LL * sms)) return false;
    const double keys = causal ? Skv - 0.5 * Sq + 0.5 * hp.rows : Skv;  // that a tile is given on average
    if (tiles > 9LL * sms) return keys <= (padded ? 256 : 320);
    return keys <= (mask_kind == FORGE_MASK_NONE || (tiles > 6LL * sms && !padded) ? 256 : 128);
}

// Head sizes above 128 run on the kernel of attn_wide.cu.  strides: of q, k, v, out, or nullptr for dense tensors.
template <bool F16>
int attn_by_head_size(const void* q, const void* k, const void* v, void* out, int B, int Hq, int Hkv, int Sq, int Skv, int D,
                      int mask_kind, const int32_t* lens, float scale, cudaStream_t s, const Strides* strides = nullptr) {
    if (D > 64 && D <= 128)
        return launch_attn<128, F16>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s, strides);
    const int sms = sm_count();
    if (sms <= 0) return FORGE_ERR_CUDA;
    if (D <= 64 && many_short_tiles(B, Hq, Hkv, Sq, Skv, mask_kind, sms))
        return launch_attn<64, F16>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s, strides);
    const Strides a = dense_strides(Hq, Sq, D), c = dense_strides(Hkv, Skv, D), dense[4] = {a, c, c, a};
    const Strides* t = strides ? strides : dense;
    long long st[4][3];
    for (int i = 0; i < 4; ++i) { st[i][0] = t[i].b; st[i][1] = t[i].h; st[i][2] = t[i].s; }
    return D <= 64 ? attn_narrow(F16, q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, st, s)
                   : attn_wide(F16, q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, st, s);
}

}  // namespace
}  // namespace forge

extern "C" int forge_attn_fused(const void* q, const void* k, const void* v, void* out,
                                int B, int Hq, int Hkv, int Sq, int Skv, int D,
                                int mask_kind, const int32_t* lens, float scale, void* stream) {
    using namespace forge;
    int st = check_attn_args(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, /*any_head_dim=*/true, 256);
    if (st != FORGE_OK) return st;
    if ((long long)Hq * B * ((Sq + 127) / 128) > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    if (!(scale >= 0.f)) return FORGE_ERR_UNSUPPORTED;  // the running maximum is taken on unscaled scores
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return attn_by_head_size<false>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s);
}

extern "C" int forge_attn_fused_f16(const void* q, const void* k, const void* v, void* out,
                                    int B, int Hq, int Hkv, int Sq, int Skv, int D,
                                    int mask_kind, const int32_t* lens, float scale, void* stream) {
    using namespace forge;
    int st = check_attn_args(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, /*any_head_dim=*/true, 256);
    if (st != FORGE_OK) return st;
    if ((long long)Hq * B * ((Sq + 127) / 128) > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    if (!(scale >= 0.f)) return FORGE_ERR_UNSUPPORTED;  // the running maximum is taken on unscaled scores
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return attn_by_head_size<true>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s);
}

extern "C" int forge_attn_fused_bias(const void* q, const void* k, const void* v, void* out,
                                     int B, int Hq, int Hkv, int Sq, int Skv, int D,
                                     int mask_kind, const int32_t* lens, const float* bias, int bias_heads,
                                     float scale, void* stream) {
    using namespace forge;
    int st = check_attn_args(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, /*any_head_dim=*/true);
    if (st != FORGE_OK) return st;
    if (!bias || (reinterpret_cast<uintptr_t>(bias) & 15u)) return FORGE_ERR_INVALID_ARG;
    if (bias_heads != 1 && bias_heads != Hq) return FORGE_ERR_INVALID_ARG;
    if ((long long)Hq * B * ((Sq + 255) / 256) > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    if (!(scale > 0.f)) return FORGE_ERR_UNSUPPORTED;  // the bias enters the kernel as bias / scale
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return D <= 64 ? launch_attn<64, false, true>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s, nullptr, bias, bias_heads)
                   : launch_attn<128, false, true>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s, nullptr, bias, bias_heads);
}

extern "C" int forge_attn_fused_strided(const void* q, const void* k, const void* v, void* out,
                                        int B, int Hq, int Hkv, int Sq, int Skv, int D,
                                        const int64_t* q_strides, const int64_t* k_strides, const int64_t* v_strides,
                                        const int64_t* out_strides, int mask_kind, const int32_t* lens, float scale,
                                        void* stream) {
    using namespace forge;
    int st = check_attn_args(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, /*any_head_dim=*/true, 256);
    if (st != FORGE_OK) return st;
    if (!q_strides || !k_strides || !v_strides || !out_strides) return FORGE_ERR_INVALID_ARG;
    if ((long long)Hq * B * ((Sq + 127) / 128) > 2147483647LL) return FORGE_ERR_UNSUPPORTED;
    if (!(scale >= 0.f)) return FORGE_ERR_UNSUPPORTED;  // the running maximum is taken on unscaled scores
    Strides str[4];
    const int64_t* in[4] = {q_strides, k_strides, v_strides, out_strides};
    for (int i = 0; i < 4; ++i) {
        str[i] = {in[i][0], in[i][1], in[i][2]};
        // rows must not overlap their own elements, and every stride must keep rows on 16-byte boundaries
        if (str[i].b <= 0 || str[i].h <= 0 || str[i].s < D) return FORGE_ERR_INVALID_ARG;
        if ((str[i].b % 8) || (str[i].h % 8) || (str[i].s % 8)) return FORGE_ERR_UNSUPPORTED;
        if (str[i].b >= (1LL << 38) || str[i].h >= (1LL << 38) || str[i].s >= (1LL << 38)) return FORGE_ERR_UNSUPPORTED;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return attn_by_head_size<false>(q, k, v, out, B, Hq, Hkv, Sq, Skv, D, mask_kind, lens, scale, s, str);
}
