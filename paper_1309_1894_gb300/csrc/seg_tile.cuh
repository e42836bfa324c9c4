// seg_tile.cuh -- one warp computes one tile of a segmented launch.
//
// A tile is a contiguous range of one problem w = RN(RN(alpha*x) + y) (paper
// Sec. 3, Fig. 1 vecwxpy).  When x, y and w share their offset modulo 32
// bytes, the warp peels the head to the 32-byte boundary, streams 256-bit
// vectors with up to MAXU vectors of x and of y per lane in flight (the
// tile's unroll U decides how many), and finishes the tail; otherwise it uses
// coalesced 8-byte accesses, kTileElems of x and of y per lane in flight.  Loads and stores are evict-first (.cs) and
// coherent, so in-place problems (w == x or w == y) are safe.
//
// One fixed-size body whose unroll is a run-time predicate serves every tile:
// a separately compiled body per (width, unroll) behind a run-time switch made
// the compiler spill registers.
#pragma once

#include "single_kernel.cuh"

namespace wx {

// Vectors of x and of y per lane in flight, at most: two (three resident blocks
// of 256 threads) or, for batches of long tiles, four (two blocks).
constexpr int kTileU = 2, kTileWideU = 4;

// How the integer-pipeline products test their operands (see ProductTest).  Three
// resident blocks leave no register for the test of the whole range: with it 1024
// segments up to 2^16 stored back to back took 34.8 us without a host's plan and
// 27.6 with one, against 34.1 and 27.3 (GB300), while the wide body takes it at no
// cost.
template <int MAXU>
constexpr ProductTest kTileTest = MAXU == kTileU ? kTestWindow : kTestVector;

__device__ __forceinline__ void tile_scalar(const double *x, const double *y, double *w,
                                            double alpha, int64_t e) {
    double xv[1], yv[1], wv[1];
    ld_vec<1, 2>(x + e, xv);
    ld_vec<1, 2>(y + e, yv);
    wxpy_vec<1>(alpha, xv, yv, wv);
    st_vec<1, 2>(w + e, wv);
}

// EMU: which operations run in the integer pipelines (fp64_emu.cuh): 0 none,
// 1 the sums of the odd positions of every 32-byte vector, 3 every product
// (with alpha's split ca).
template <int EMU, int MAXU>
__device__ __forceinline__ void tile_body4(const double *x, const double *y, double *w,
                                           double alpha, const MulCoef &ca, int64_t nch, int lane,
                                           int U) {
    U = min(U, MAXU);
    const int64_t step = 32 * U;
    for (int64_t c0 = lane; c0 < nch; c0 += step) {
        double xv[MAXU][4], yv[MAXU][4], wv[MAXU][4];
#pragma unroll
        for (int u = 0; u < MAXU; ++u) {
            const int64_t c = c0 + 32 * u;
            if (u < U && c < nch) {
                ld_vec<4, 2>(x + c * 4, xv[u]);
                ld_vec<4, 2>(y + c * 4, yv[u]);
            }
        }
#pragma unroll
        for (int u = 0; u < MAXU; ++u) {
            const int64_t c = c0 + 32 * u;
            if (u < U && c < nch) {
                wxpy_vec_emu<4, EMU, kTileTest<MAXU>>(alpha, ca, xv[u], yv[u], wv[u], 0);
                st_vec<4, 2>(w + c * 4, wv[u]);
            }
        }
    }
}

// The same for pointers whose offsets differ modulo 32 bytes: single elements,
// a warp's accesses contiguous.  One element per lane at a time waited out the
// memory latency for every 32 elements: a batch of 2048 segments up to 2^16
// elements (1.2e7 in all) with differing offsets took 169 us on GB300, 52 with eight.
constexpr int kTileElems = 8;

template <int EMU>
__device__ __forceinline__ void tile_elements(const double *x, const double *y, double *w,
                                              double alpha, const MulCoef &ca, int64_t len,
                                              int lane) {
    for (int64_t e0 = lane; e0 < len; e0 += 32 * kTileElems) {
        double xv[kTileElems / 4][4], yv[kTileElems / 4][4];
#pragma unroll
        for (int u = 0; u < kTileElems; ++u) {
            double a[1] = {1.0}, b[1] = {1.0};  // past the end: a plain product, not stored
            if (e0 + 32 * u < len) {
                ld_vec<1, 2>(x + e0 + 32 * u, a);
                ld_vec<1, 2>(y + e0 + 32 * u, b);
            }
            xv[u / 4][u % 4] = a[0];
            yv[u / 4][u % 4] = b[0];
        }
#pragma unroll
        for (int g = 0; g < kTileElems / 4; ++g) {
            double wv[4];
            wxpy_vec_emu<4, EMU, kTileTest<kTileU>>(alpha, ca, xv[g], yv[g], wv, 0);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int64_t e = e0 + 32 * (4 * g + u);
                const double r[1] = {wv[u]};
                if (e < len) st_vec<1, 2>(w + e, r);
            }
        }
    }
}

// The whole tile [x, x+len) by the calling warp (lane = thread index mod 32).
template <int EMU, int MAXU = kTileU>
__device__ __forceinline__ void tile_wxpy(const double *x, const double *y, double *w,
                                          double alpha, int64_t len, int lane, int U) {
    MulCoef ca{};
    if constexpr (EMU == 3) ca = mul_coef_of((uint64_t)__double_as_longlong(alpha));
    const uintptr_t ax = (uintptr_t)x, ay = (uintptr_t)y, aw = (uintptr_t)w;
    if ((((ax ^ aw) | (ay ^ aw)) & 31u) == 0) {
        const int64_t head = min(len, (int64_t)((4 - (int)((aw >> 3) & 3)) & 3));
        const int64_t nch = (len - head) / 4;
        const int64_t body_end = head + nch * 4;
        if (lane < head) tile_scalar(x, y, w, alpha, lane);
        if (lane >= 4 && body_end + (lane - 4) < len)
            tile_scalar(x, y, w, alpha, body_end + (lane - 4));
        tile_body4<EMU, MAXU>(x + head, y + head, w + head, alpha, ca, nch, lane, U);
    } else {
        tile_elements<EMU>(x, y, w, alpha, ca, len, lane);
    }
}

}  // namespace wx
