// How the forward cuts a batch into tiles and its warps walk them: without CUDA
// types, so that a host compiler takes it too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define PSS_HD __host__ __device__ __forceinline__
#else
#define PSS_HD inline
#endif

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

// The tiles (table t, range r of wb bags) of one warp: every nwarps-th in the order
// of the bags (number r * T + t) or of the tables (t * tpt + r), reached without
// divisions.  32-bit numbers, below kMaxTiles (unsigned: a step or two past the
// last tile stay in range).
constexpr int64_t kMaxTiles = int64_t(1) << 31;

struct TileWalk {
    uint32_t T, tpt;              // tables, tiles per table
    uint32_t step_t, step_r;
    int64_t step_o, wrap_o;       // the same as distances in the offsets
    bool by_table;
    PSS_HD TileWalk(uint32_t nwarps, uint32_t T_, uint32_t tpt_, int64_t B, int wb, bool by_table_)
        : T(T_), tpt(tpt_), by_table(by_table_) {
        const uint32_t inner = by_table ? tpt : T;
        const uint32_t step_out = nwarps / inner, step_in = nwarps - step_out * inner;
        step_t = by_table ? step_out : step_in;
        step_r = by_table ? step_in : step_out;
        step_o = (int64_t)step_t * B + (int64_t)step_r * wb;
        wrap_o = by_table ? B - (int64_t)tpt * wb : wb - (int64_t)T * B;
    }
    PSS_HD void first(uint32_t tile, uint32_t& t, uint32_t& r) const {
        const uint32_t inner = by_table ? tpt : T, out = tile / inner;
        t = by_table ? out : tile - out * inner;
        r = by_table ? tile - out * inner : out;
    }
    PSS_HD bool inside(uint32_t t, uint32_t r) const { return t < T && r < tpt; }
    // To the next tile; returns the distance in the offsets.
    PSS_HD int64_t advance(uint32_t& t, uint32_t& r) const {
        t += step_t;
        r += step_r;
        if (by_table ? r < tpt : t < T) return step_o;
        if (by_table) {
            r -= tpt;
            ++t;
        } else {
            t -= T;
            ++r;
        }
        return step_o + wrap_o;
    }
};

}  // namespace pss
