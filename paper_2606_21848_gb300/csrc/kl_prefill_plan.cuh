// Launch layout of the chunked prefill, chosen on the host from sizes alone (plain C++, no CUDA).
#pragma once

#include <stdint.h>

namespace kl {

struct PrefillPlan {
    int hp;    // heads of a value head's group in a block of 128 rows
    int rpb;   // query rows per block: 128 / hp
    int cs;    // CTAs of the cluster that splits a block's cache tiles: 1, 2, 4 or 8
};

constexpr int kPrefillRows = 128;          // rows of a block
constexpr int kPrefillTile = 128;          // cache rows of a tile
constexpr int64_t kMaxGridZ = 65535;       // blocks of query rows are the grid's z extent

// B sequences, Hkv value heads of G query heads, chunks of at most max_q rows, tables of max_tokens
// tokens, sms multiprocessors.
inline PrefillPlan plan_prefill(int B, int Hkv, int G, int max_q, int64_t max_tokens, bool wr_per_qh,
                                int sms) {
    PrefillPlan p{1, kPrefillRows, 1};
    const auto row_blocks = [&](int hp) {
        return ((int64_t)max_q + kPrefillRows / hp - 1) / (kPrefillRows / hp);
    };
    const auto blocks_of = [&](int hp) { return (int64_t)((G + hp - 1) / hp) * row_blocks(hp); };
    // Heads per block: a block's 128 rows hold hp heads of a group (which read the same tiles),
    // 128 / hp query rows each; the fewest blocks, and the fewest heads among equals. One W^R per
    // query head: one head per block, which has one routing matrix. A chunk so long that the row
    // blocks of hp heads would not fit the grid (131073 rows at 64 heads, 1.05 M at 8) takes fewer
    // heads; one head per block fits every length that the entry point accepts.
    if (!wr_per_qh)
        for (int hp = 2; hp <= G && hp <= 64; ++hp)
            if (blocks_of(hp) < blocks_of(p.hp) && row_blocks(hp) <= kMaxGridZ) p.hp = hp;
    p.rpb = kPrefillRows / p.hp;
    // CTAs per block: while the blocks leave half of the SMs idle, clusters of 2, 4 or 8 CTAs
    // split a block's tiles (at least two tiles each at the longest length). A cluster's CTAs sit
    // in one GPC, which leaves some of its SMs over: pairs fill all of them, clusters of 4 and 8
    // are counted on for 27/32. (6 sequences of 46000 tokens, 112-token chunks, 12 heads, 72
    // blocks: 379 us, in pairs 207.)
    const int64_t blocks = blocks_of(p.hp) * Hkv * B;
    const int64_t tiles = (max_tokens + kPrefillTile - 1) / kPrefillTile;
    while (p.cs < 8 && p.cs * 4 <= tiles && blocks * p.cs * 2 * 32 <= (int64_t)sms * (p.cs == 1 ? 32 : 27))
        p.cs *= 2;
    return p;
}

}  // namespace kl
