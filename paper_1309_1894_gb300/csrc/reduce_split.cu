// reduce_split.cu -- the fused reductions on few tiles (a tile over a cluster
// of eight blocks) and the tree over the tile sums of every form.
//
// The update is the paper's (Sec. 3, Fig. 1); the tree is the one of
// reduce.cu.  Element i of a tile has bits 12..10 = row k, 9..7 = column c,
// 6..0 = position in the column.  The tree reduces bits from the top down, so
// a column is independent of the others until bits 12..10 are done: block c of
// a cluster takes column c, 1024 elements, warp k of it row k, one 32-byte
// vector of every operand per lane.  The rows meet in shared memory (bits
// 12..10, one position per thread), the eight columns in the first block's
// shared memory (bits 9..7), and one warp sums the 128 positions.
//
// What bounds it: the latency of one pass.  A tile in one block is 8192
// elements behind one SM's FP64 pipeline (two sums each, 1.7 per clock: 5 us)
// and eight dependent loads per thread; here a block holds 1024 elements and
// every thread loads once.
#include "cluster.cuh"
#include "reduce_common.cuh"
#include "single_kernel.cuh"

namespace wx {
namespace {

constexpr int kColumns = 8;         // blocks of a cluster
constexpr int kSplitThreads = 256;  // eight rows, one warp each

// Stores v at `p` (an address of this block's shared memory) in block 0 of the cluster.
__device__ __forceinline__ void st_first_block(double *p, double v) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, 0;"
                 : "=r"(remote)
                 : "r"((uint32_t)__cvta_generic_to_shared(p)));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

// The terms of one row of C neighbouring columns (128 C elements from `base`)
// into row[0 .. 128 C - 1]; w stored, +0 terms past n.  VEC: lane l takes
// elements 4l .. 4l + 3 of a column as one 32-byte vector of every operand,
// where they are all there.  Else lane l takes elements l + 32 q, so that the
// 8-byte accesses of a warp are contiguous.  Every load is issued before the
// first store.  x outside the integer products' range (zeros, say) is told before
// the update's sum: no tile here has a next one to take with other products.  Every
// seventh element zero, norm2 at 2^21 elements 21.4 us against 29.6, with differing
// offsets at 2^23 73.8 against 102, dot there 80.1 against 105; other data within
// 1.5 % either way.  dot on vectors of two columns has no register for it (2^21
// elements 20.4 us on other data against 19.0).
template <int KIND, bool VEC, bool EMU, int C>
__device__ __forceinline__ void row_terms(const ReduceArgs &a, int64_t base, int lane, double *row) {
    if constexpr (VEC) {
        if (base + 128 * C <= a.n) {
            double x[C][4], y[C][4], z[KIND == 1 ? C : 1][4];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int64_t i = base + 128 * c + 4 * lane;
                ld4(a.x + i, x[c]);
                ld4(a.y + i, y[c]);
                if constexpr (KIND == 1) ld4(a.z + i, z[c]);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                double w[4], t[4];
                bool left;
                elements4<KIND, EMU ? kInteger : kFp64, KIND == 0 || C == 1>(
                    a, x[c], y[c], z[KIND == 1 ? c : 0], w, t, left);
                st4(a.w + base + 128 * c + 4 * lane, w);
                double2 *r = reinterpret_cast<double2 *>(row + 128 * c + 4 * lane);
                r[0] = make_double2(t[0], t[1]);
                r[1] = make_double2(t[2], t[3]);
            }
            return;
        }
    }
    double x[4 * C], y[4 * C], z[KIND == 1 ? 4 * C : 1];
#pragma unroll
    for (int q = 0; q < 4 * C; ++q) {
        const int64_t i = base + lane + 32 * q;
        if (i < a.n) {
            x[q] = a.x[i];
            y[q] = a.y[i];
            if constexpr (KIND == 1) z[q] = a.z[i];
        }
    }
#pragma unroll
    for (int q = 0; q < 4 * C; ++q) {
        const int64_t i = base + lane + 32 * q;
        double t = 0.0;
        if (i < a.n) {
            double w;
            bool left;
            element<KIND, EMU && !VEC ? kIntegerEach : kFp64>(a, x[q], y[q], KIND == 1 ? z[q] : 0.0,
                                                               w, t, left);
            a.w[i] = w;
        }
        row[lane + 32 * q] = t;
    }
}

template <int KIND, bool VEC, int C>
__global__ void __cluster_dims__(kColumns / C, 1, 1) __launch_bounds__(kSplitThreads)
    wxpy_reduce_split_kernel(const ReduceArgs a) {
    constexpr int kBlocks = kColumns / C;  // of a cluster
    __shared__ __align__(16) double rows[8][128 * C];
    __shared__ double cols[kColumns][128];  // used in the cluster's first block
    const int t = threadIdx.x, lane = t & 31, k = t >> 5;
    const int part = blockIdx.x & (kBlocks - 1);
    const int64_t tile = blockIdx.x / kBlocks;
    const int64_t base = tile * kTile + 1024 * k + 128 * C * part;
    cluster_arrive();  // the first block's shared memory may be written once all have started
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const int64_t i = base + 128 * c + 4 * lane;
        if (i < a.n) {
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.x + i));
            asm volatile("prefetch.global.L2 [%0];" ::"l"(a.y + i));
            if constexpr (KIND == 1) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.z + i));
        }
    }
    pdl_enter();
    // the pipe choice rotates over the tiles
    if ((((unsigned)tile * 7u) & 15u) < (unsigned)a.mul_sixteenths)
        row_terms<KIND, VEC, true, C>(a, base, lane, rows[k]);
    else
        row_terms<KIND, VEC, false, C>(a, base, lane, rows[k]);
    __syncthreads();
    cluster_wait();
    if (t < 128 * C)  // bits 12..10
        st_first_block(&cols[0][128 * C * part + t], tree8<128 * C>(&rows[0][t]));
    cluster_arrive();
    cluster_wait();
    if (part != 0) return;
    if (t < 128) rows[0][t] = tree8<128>(&cols[0][t]);  // bits 9..7
    __syncthreads();
    if (t < 32) {
        const double s = column_sum(rows[0], lane);
        if (lane == 0) *(a.ntiles == 1 ? a.result : a.partial + tile) = s;
    }
}

// ---- the tree over the tile sums -------------------------------------------------
//
// One block.  Thread t takes the sums t + 1024 k, so the top levels run in the
// thread with all its loads in flight at once; the next ones, down to 32
// values, through shared memory, the last by shuffles.  More than
// kFinalInThread of them are first halved in place, level by level.  It is
// launched with programmatic serialisation and waits for the form's kernel by
// griddepcontrol, so its launch overlaps that kernel; a ticket that elects the
// last block instead would need the workspace cleared before every call.

constexpr int kFinalThreads = 1024;
constexpr int kFinalPerThread = 16;
constexpr int64_t kFinalInThread = (int64_t)kFinalThreads * kFinalPerThread;

__global__ void __launch_bounds__(kFinalThreads, 1) wxpy_reduce_final_kernel(const ReduceArgs a) {
    __shared__ double sm[kFinalThreads];
    const int t = threadIdx.x;
    pdl_enter();
    int64_t p = a.padded_tiles, have = a.ntiles;  // +0 from `have` on
    for (; p > kFinalInThread; p /= 2) {
        const int64_t half = p / 2;
        for (int64_t i = t; i < half; i += kFinalThreads) {
            const double hi = i + half < have ? __ldcg(a.partial + i + half) : 0.0;
            a.partial[i] = __dadd_rn(i < have ? __ldcg(a.partial + i) : 0.0, hi);
        }
        have = half;
        __syncthreads();
    }
    double e[kFinalPerThread];
#pragma unroll
    for (int k = 0; k < kFinalPerThread; ++k) {
        const int64_t i = t + (int64_t)kFinalThreads * k;
        e[k] = i < have ? __ldcg(a.partial + i) : 0.0;
    }
#pragma unroll
    for (int s = kFinalPerThread / 2; s >= 1; s /= 2) {
        if (p >= 2ll * s * kFinalThreads) {  // a level the tree has: no sum with padding beyond it
#pragma unroll
            for (int k = 0; k < s; ++k) e[k] = __dadd_rn(e[k], e[k + s]);
        }
    }
    double v = e[0];
    const int m = (int)(p < kFinalThreads ? p : kFinalThreads);
    for (int s = m / 2; s >= 32; s /= 2) {
        if (t < 2 * s) sm[t] = v;
        __syncthreads();
        if (t < s) v = __dadd_rn(v, sm[t + s]);
        __syncthreads();
    }
    if (t < 32) {
#pragma unroll
        for (int sh = 16; sh >= 1; sh >>= 1) {
            const double u = __shfl_down_sync(0xffffffffu, v, sh);
            if (2 * sh <= m) v = __dadd_rn(v, u);
        }
        if (t == 0) *a.result = v;
    }
}

}  // namespace

// Tiles up to which a block takes one column (clusters of eight): beyond, its
// blocks no longer all fit at once, and two columns per block (clusters of
// four) are faster.  norm2 / dot, us, one against two columns: 400000 elements
// (49 tiles) 6.2 / 6.5 against 6.8 / 7.3, 10^6 (123) 10.3 / 12.0 against
// 10.0 / 11.0, 2^21 (256) 18.1 / 19.1 against 16.7 / 18.2.
constexpr int64_t kOneColumnTiles = 76;

template <int KIND, bool VEC, int C>
static cudaError_t launch_split(const ReduceArgs &a, cudaStream_t s) {
    return launch_pdl(&wxpy_reduce_split_kernel<KIND, VEC, C>, (unsigned)(a.ntiles * (kColumns / C)),
                      kSplitThreads, s, a);
}

cudaError_t launch_reduce_split(int kind, bool vec, const ReduceArgs &a, cudaStream_t s) {
    const bool one = a.ntiles <= kOneColumnTiles;
    if (kind == 0)
        return vec ? (one ? launch_split<0, true, 1>(a, s) : launch_split<0, true, 2>(a, s))
                   : (one ? launch_split<0, false, 1>(a, s) : launch_split<0, false, 2>(a, s));
    // dot on single elements holds three operands of two columns in 72 registers:
    // one column is faster throughout (2^21 elements 19.9 against 21.4 us)
    return vec ? (one ? launch_split<1, true, 1>(a, s) : launch_split<1, true, 2>(a, s))
               : launch_split<1, false, 1>(a, s);
}

cudaError_t launch_reduce_final(const ReduceArgs &a, cudaStream_t s) {
    const int64_t p = a.padded_tiles;
    const unsigned threads = (unsigned)(p < 32 ? 32 : p < kFinalThreads ? p : kFinalThreads);
    return launch_pdl(&wxpy_reduce_final_kernel, 1u, threads, s, a);
}

}  // namespace wx
