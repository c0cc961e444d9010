// How the forward cuts a batch into tiles: host rules without CUDA types.
#pragma once

#include <cstdint>

namespace pss {

constexpr int kWarpPairs = 512;   // staged pairs per warp and round
constexpr int kMaxTileBags = 32;  // bags per tile at most: one lane each

// Bags per tile of the forward: a multiple of the lane groups (and of 4), at
// most kMaxTileBags, kWarpPairs staged pairs, and 16 bags or 4 per lane group,
// chosen so that the warps' rounds of tiles waste least: rounds * (wb + 8) is
// smallest, a tile's fixed work being about that of 8 bags.  Measured on GB300,
// us per forward at 4, 8, 12, 16, 24 and 32 bags: Criteo-TB shape 227, 158, 150,
// 153, 156, 156; multi-hot 326, 310, 303, 294, 298, 314; 16-float rows (batch
// 16384, 8 lane groups) 36, 25, 18, 14, 11, 9.6.
inline int tile_bags(int64_t T, int J, int log2gs, int64_t rows, int64_t warps) {
    const int ng = 32 >> log2gs;
    const int step = ng > 4 ? ng : 4;
    int best = step;
    int64_t best_cost = INT64_MAX;
    const int some = 4 * ng > 16 ? 4 * ng : 16;
    const int most = some < kMaxTileBags ? some : kMaxTileBags;
    for (int wb = step; wb <= most; wb += step) {
        if (wb > step && wb * J > kWarpPairs) break;
        const int64_t tiles = T * ((rows + wb - 1) / wb);
        const int64_t cost = ((tiles + warps - 1) / warps) * (wb + 8);
        if (cost <= best_cost) {
            best_cost = cost;
            best = wb;
        }
    }
    return best;
}

}  // namespace pss
