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

// CTAs that share a row in the SiLU quantiser (a cluster; 1: one CTA per row), by rows and channels: a cluster's start and two
// barriers pay only where a row is long and the rows are few.  Measured on B200 on both sides of each line, time with the
// cluster over time with one CTA per row, alone and behind two sizes of the projection: 16 rows of 4096 channels 1.05 (alone),
// of 5120 0.84 to 0.94; 24 of 6144 0.89, 1.23 and 1.17, of 8192 0.84 to 0.99; 48 of 4096 0.99 to 1.06, of 5120 0.82 to 0.93; 64 of
// 5120 1.06 to 1.10, of 8192 0.89 to 1.00; 96 of 8192 0.98 to 1.01, of 12288 0.91 to 0.97; 160 of 6144 0.93 to 1.03, of 8192 0.80 to
// 0.99; 200 of 6144 1.18 alone and 0.95 to 0.98 behind, of 8192 1.02 and 0.89 to 0.92; 300 of 6144 0.99 to 1.09, of 10240 0.89
// to 0.97; 700 of 10240 1.03 to 1.11.  On short rows it is up to twice as long (256 of 512 alone: 4.9 and 2.5 us).
inline int silu_cluster_ctas(int M, int K) {
    struct Line { int rows, min_channels, ctas; };
    constexpr Line LINES[] = {{16, 5120, 8}, {32, 8192, 8}, {48, 5120, 8}, {64, 8192, 8}, {128, 12288, 8}, {160, 8192, 8}, {256, 8192, 4}, {600, 10240, 2}};
    for (const Line& l : LINES)
        if (M <= l.rows) return K >= l.min_channels ? l.ctas : 1;
    return 1;
}

}  // namespace w4a8
