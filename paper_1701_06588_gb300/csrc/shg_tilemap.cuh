// Which tile a warp takes: 32-pair tiles of a plan's class chunks (TileMap), and the warps of a static launch.
#pragma once

#include "shg_internal.h"

namespace shg {

// Index of a warp among those of a launch with one tile per warp.  From the block and the warp within it: the index of the
// thread passes 2^32 with 2^27 tiles, and a plan of 2^30 pairs with eight lanes each has 2^28.
__host__ __device__ constexpr int launch_warp(unsigned block, unsigned threads, unsigned thread)
{
    return (int)(block * (threads >> 5) + (thread >> 5));
}

// position in the sorted list of the pair of `lane` in 32-pair tile t, and its class; -1 for a lane past the chunk's end
__device__ __forceinline__ int map_pair(const TileMap &m, int t, int lane, int &cls)
{
    int lo = 0, hi = kNClass;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (m.tile[mid] <= t) lo = mid;
        else hi = mid;
    }
    cls = m.cls[lo];
    const int q = m.pair[lo] + (t - m.tile[lo]) * kTile + lane;
    return q < m.pair[lo + 1] ? q : -1;
}

}  // namespace shg
