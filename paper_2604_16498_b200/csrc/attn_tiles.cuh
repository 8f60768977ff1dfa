// How the query rows of grouped heads share a 128-row tile (attn_bf16.cu, attn_wide.cu).
#pragma once

namespace forge {

// A tile holds `rows` consecutive query rows of each of `pack` query heads of one KV group: row h * rows + i of the tile is query
// row q0 + i of the h-th of them.
struct HeadPack {
    int pack, rows;  // pack divides the heads per KV head; pack * rows <= 128
};

// The division of G = Hq / Hkv heads and Sq rows that computes the fewest scores: tiles times the keys that a tile's rows are
// given on average.  With a causal mask that is the mean visible length plus half of the rows (a tile goes on to the last key of
// its last row) and half of a 64-key step, so more heads and fewer rows of each win where the tiles are equally many; without one,
// fewer heads do.  in_pairs: two consecutive tiles are an item, and one without a second costs a little more than half.
// Against one head per tile: 3 x 28/4 heads x 777 x 1801, D = 128, 62.8 -> 49.6 us (49 tiles of a KV head and batch entry become
// 44), 64 x 16/4 x 64 15.6 -> 12.8, 4 x 32/8 x 2048 causal 130.6 -> 128.0 (3 % fewer scores above the diagonal).
inline HeadPack choose_pack(int G, int Sq, int Skv, bool causal, bool in_pairs) {
    HeadPack best = {1, 128};
    double best_cost = 0;
    for (int pack = 1; pack <= 16 && pack <= G; ++pack) {
        if (G % pack) continue;
        const int rows = 128 / pack;
        const double keys = causal ? Skv - 0.5 * Sq + 0.5 * rows + 32 : Skv;
        const int tiles = (Sq + rows - 1) / rows;
        const double cost = (G / pack) * (tiles + (in_pairs && tiles % 2 ? 0.1 : 0.)) * keys;
        if (pack == 1 || (causal ? cost <= best_cost : cost < best_cost)) { best_cost = cost; best = {pack, rows}; }
    }
    return best;
}

}  // namespace forge
