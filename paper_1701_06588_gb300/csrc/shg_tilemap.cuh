// 32-pair tiles of a plan's class chunks (TileMap).
#pragma once

#include "shg_internal.h"

namespace shg {

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
