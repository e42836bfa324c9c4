// seg_search.cuh -- the tiles of a segmented launch without a tile list: a plan
// entry per segment, and warps that find their tile's segment in it.
#pragma once

#include "internal.h"
#include "seg_tile.cuh"

namespace wx {

// One segment: its first tile in the launch's numbering, the elements its tiles
// cover, and its tile length with log2 of the unroll in the top bits.
struct SegPlan {
    int64_t first_tile;
    int64_t n;
    uint32_t len_ul;
    uint32_t pad;
    __host__ __device__ int64_t tile_len() const { return (int64_t)(len_ul & kLenMask); }
};

__host__ __device__ inline SegPlan seg_plan_of(int64_t n, int64_t first_tile, int64_t tile_len,
                                               int unroll_log2) {
    return SegPlan{first_tile, n, (uint32_t)tile_len | (uint32_t)unroll_log2 << 30, 0u};
}

// The segment of tile t: the largest s in [lo, count) with plan[s].first_tile <= t,
// by the whole warp, 32 probes at a time; plan[lo].first_tile <= t.
__device__ __forceinline__ int64_t find_segment(const SegPlan *plan, int64_t count, int64_t t,
                                                int64_t lo, int lane) {
    int64_t hi = count;
    while (hi - lo > 1) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t i = lo + lane * step;
        const unsigned below = __ballot_sync(0xffffffffu, i < hi && plan[i].first_tile <= t);
        lo += (int64_t)(31 - __clz(below)) * step;  // the probes ascend; lane 0's is below
        hi = min(hi, lo + step);
    }
    return lo;
}

// One tile; one that would pass the n of the descriptor it reads is skipped.
template <int EMU, int MAXU>
__device__ __forceinline__ void run_plan_tile(const wxpy_desc &d, const SegPlan &sp, int64_t t,
                                              int lane) {
    const int64_t T = sp.tile_len(), begin = (t - sp.first_tile) * T;
    const int64_t len = min(T, sp.n - begin);
    if (len > 0 && begin + len <= d.n)
        tile_wxpy<EMU, MAXU>(d.x + begin, d.y + begin, d.w + begin, d.alpha, len, lane,
                             1 << (sp.len_ul >> 30));
}

// Every tile of a plan of `count` segments (plan[count].first_tile: the tile
// count).  Where most segments are one tile, a warp takes a run of neighbouring
// tiles, searches once and walks the plan: the search is most of a short tile's
// time (40000 segments up to 1024 elements 85 us against 115 on GB300).  Else
// warp k takes tiles k, k + W, .. and searches for each, so that the warps of an
// SM work on neighbouring memory (4096 segments up to 2^20: 1141 us against 1210).
template <int EMU, int MAXU>
__device__ __forceinline__ void run_plan_tiles(const wxpy_desc *table, const SegPlan *plan,
                                               int64_t count) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t ntiles = plan[count].first_tile;
    const int64_t used = min(ntiles, nwarps);  // with few tiles the last blocks have none
    if (warp >= used) return;
    const bool runs = ntiles < 2 * count;
    int64_t t = runs ? ntiles * warp / used : warp;
    const int64_t end = runs ? ntiles * (warp + 1) / used : ntiles, step = runs ? 1 : nwarps;
    for (int64_t s = 0; t < end; t += step) {
        if (s == 0 || !runs) s = find_segment(plan, count, t, s, lane);
        while (plan[s + 1].first_tile <= t) ++s;
        run_plan_tile<EMU, MAXU>(table[s], plan[s], t, lane);
    }
}

}  // namespace wx
