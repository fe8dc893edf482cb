// Rules of the dispatch that depend on sizes alone (plain C++: they are tested on the CPU).
#pragma once

namespace w4a8 {

// Token-tile height (208, 128 or 64 rows) of the per-channel form, whose tiles of every height run in
// gemm_tcgen05_kernel: whole tiles in rounds over the SMs, at a cost per round and group of which only the ratios matter.
// Measured on B200 over 13 layers at 65 to 3000 tokens, every height forced: this choice is within 5 % of the best height but for
// 512 -> 8192 at 80 and 300 tokens (6.5 and 8.3 us, 5.7 and 7.7) and 5120 -> 27648 at 448 (83.2, 74.2).  Priced like the grouped
// form, whose 64-row tiles are those of gemm_tcshort.cu, it fell for a round more of 64-row tiles: 5120 -> 7168 at 300
// tokens 29.2 us (208 rows: 20.4), 12288 -> 4096 at 513 63.5 (41.2), 4096 -> 24576 at 160 42.1 (27.6).
inline int per_channel_tile_height(int M, int n_tiles, int groups, int sms) {
    constexpr int HEIGHTS[3] = {208, 128, 64};
    constexpr long FIXED = 4000, GROUP_COST[3] = {650, 540, 440};
    int best = 64;
    long best_cost = -1;
    for (int i = 0; i < 3; ++i) {
        if (i < 2 && M <= HEIGHTS[i + 1]) continue;                 // the next height down already covers M in one tile
        const long tiles = (long)((M + HEIGHTS[i] - 1) / HEIGHTS[i]) * n_tiles;
        const long cost = FIXED + (tiles + sms - 1) / sms * GROUP_COST[i] * groups;
        if (best_cost < 0 || cost < best_cost) {                    // ties: the taller tile
            best_cost = cost;
            best = HEIGHTS[i];
        }
    }
    return best;
}

}  // namespace w4a8
