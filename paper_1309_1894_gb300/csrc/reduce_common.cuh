// reduce_common.cuh -- what the fused reductions' kernel forms share: the
// tile of the fixed summation tree, the argument block, the per-element
// arithmetic (w = RN(RN(alpha*x) + y) of paper Sec. 3, Fig. 1, then the
// term RN(w*w) or RN(w*z)), the integer-pipeline tree sum of non-negative
// values, the 32-byte accesses, and the end of a tile's tree.
// Included by reduce.cu (register-loaded and staged forms), reduce_warp.cu
// (warp-tiled form) and reduce_split.cu (a tile over a cluster of blocks, and
// the tree over the tile sums); everything is internal to each.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "fp64_addpos.cuh"
#include "fp64_emu.cuh"
#include "fp64_mul.cuh"
#include "internal.h"

namespace wx {

constexpr int kTile = 8192;
constexpr int64_t kHeaderBytes = 256;  // before the tile sums in the workspace

struct ReduceArgs {
    const double *x, *y, *z;  // z: dot only
    double *w;
    double *result;
    double *partial;  // the tile sums: padded_tiles slots
    int64_t n, ntiles, padded_tiles;
    double alpha;
    MulCoef ca;
    int mul_sixteenths;
    int shift;           // elements w starts past a 32-byte boundary (0..3)
    int64_t drop_chunk;  // staged path: the producer stops before this chunk (-1: never)
};

// The warp-tiled form (reduce_warp.cu): launches the kernel of `shape`
// (0: two rows per load group, five blocks of 128 threads per SM; 1: four
// rows, four blocks; 2: four rows, three blocks) for kind 0 (norm2, `suml`
// leading tree levels 0..6 in the integer pipelines) or 1 (dot, suml 0) on
// 32-byte co-aligned pointers.
cudaError_t launch_reduce_warp(int kind, int suml, int shape, const ReduceArgs &a,
                               const DeviceProps *dp, cudaStream_t s);

namespace {

__device__ __forceinline__ uint64_t bits_of(double v) { return (uint64_t)__double_as_longlong(v); }
__device__ __forceinline__ double double_of(uint64_t b) { return __longlong_as_double((long long)b); }

static __device__ __noinline__ uint64_t add_rn_hw_bits(uint64_t ua, uint64_t ub) {
    return bits_of(__dadd_rn(double_of(ua), double_of(ub)));
}

// RN(a + b) of two sums of squares (non-negative): the integer-pipeline sum
// when INT, else the FP64 instruction.
template <bool INT>
__device__ __forceinline__ double tree_add(double a, double b) {
    if constexpr (INT) {
        const uint64_t ua = opaque_bits(a), ub = opaque_bits(b);
        bool slow = false;
        uint64_t r = add_pos_core(ua, ub, slow);
        if (slow) r = add_rn_hw_bits(ua, ub);  // out of line
        return double_of(r);
    } else {
        return __dadd_rn(a, b);
    }
}

// w and the term of one element with both products on the FP64 pipeline, as
// bit patterns (w in x, the term in y of the result).  Out of line: it runs
// only when an integer-pipeline product left its fast path, and inlined it
// would be issued, predicated off, for every element.
template <int KIND>
static __device__ __noinline__ ulonglong2 element_hw_bits(uint64_t alpha, uint64_t x, uint64_t y,
                                                          uint64_t z) {
    const double w = __dadd_rn(__dmul_rn(double_of(alpha), double_of(x)), double_of(y));
    const double t = __dmul_rn(w, KIND == 0 ? w : double_of(z));
    return make_ulonglong2(bits_of(w), bits_of(t));
}

static __device__ __noinline__ uint64_t mul_hw_bits(uint64_t ua, uint64_t ub) {
    return bits_of(__dmul_rn(double_of(ua), double_of(ub)));
}

// Where an element's two products run: both on the FP64 pipeline, both in the
// integer pipelines, or the term's alone there.
enum Products : int { kFp64, kInteger, kIntegerEach, kTermInteger };

// w and the term of one element.  kInteger: one fallback test for the element,
// and `left` set when it left the fast path.  At n = 2^26 (GB300) products with
// one test run norm2 / dot at 0.75 / 0.89 of the measured peak, against
// 0.72 / 0.84 with the fully checked products and a test for each.  kIntegerEach:
// a test for each all the same, so that x outside the range (zeros, say) pays for
// no second sum, and `left` set by the term's alone.
template <int KIND, int MODE>
__device__ __forceinline__ void element(const ReduceArgs &a, double x, double y, double z,
                                        double &w, double &t, bool &left) {
    if constexpr (MODE == kTermInteger || MODE == kIntegerEach) {
        if constexpr (MODE == kTermInteger) {
            w = __dadd_rn(__dmul_rn(a.alpha, x), y);
        } else {
            uint32_t far = 0;
            uint64_t pb = mul_rn_range(a.ca, bits_of(x), far);
            if (far >= a.ca.span) pb = mul_hw_bits(bits_of(a.alpha), bits_of(x));
            w = __dadd_rn(double_of(pb), y);
        }
        const uint64_t wb = opaque_bits(w), zb = KIND == 0 ? wb : bits_of(z);
        bool slow = false;
        uint64_t tb = KIND == 0 ? sqr_rn_core(wb, slow) : mul_rn_quick2(wb, zb, slow);
        if (slow) {
            tb = mul_hw_bits(wb, zb);
            left = true;
        }
        t = double_of(tb);
    } else if constexpr (MODE == kInteger) {
        uint32_t far = 0;
        bool slow = false;
        w = __dadd_rn(double_of(mul_rn_range(a.ca, bits_of(x), far)), y);
        const uint64_t wb = opaque_bits(w);
        t = double_of(KIND == 0 ? sqr_rn_core(wb, slow) : mul_rn_quick2(wb, bits_of(z), slow));
        if (slow || far >= a.ca.span) {
            const ulonglong2 r =
                element_hw_bits<KIND>(bits_of(a.alpha), bits_of(x), bits_of(y), bits_of(z));
            w = double_of(r.x);
            t = double_of(r.y);
            left = true;
        }
    } else {
        w = __dadd_rn(__dmul_rn(a.alpha, x), y);
        t = __dmul_rn(w, KIND == 0 ? w : z);
    }
}

template <int KIND, bool EMU>
__device__ __forceinline__ void element(const ReduceArgs &a, double x, double y, double z,
                                        double &w, double &t) {
    bool left;
    element<KIND, EMU ? kInteger : kFp64>(a, x, y, z, w, t, left);
}

// w and the terms of four elements.  EARLY (of kInteger): the range of the four x
// is tested before their products, so that data outside it (zeros, say) pays for
// no second update sum, and `left` is set by the terms' products alone.  It costs
// norm2 on data inside 2 % at 2^25 elements and 4 % at 2^26, dot nothing.
template <int KIND, int MODE, bool EARLY>
__device__ __forceinline__ void elements4(const ReduceArgs &a, const double (&x)[4],
                                          const double (&y)[4], const double (&z)[4],
                                          double (&w)[4], double (&t)[4], bool &left) {
    if constexpr (MODE == kInteger && EARLY) {
        uint32_t far = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) far = max(far, mul_distance(a.ca, bits_of(x[q])));
        uint64_t pb[4];
        if (far >= a.ca.span) {
#pragma unroll
            for (int q = 0; q < 4; ++q) pb[q] = mul_hw_bits(bits_of(a.alpha), bits_of(x[q]));
        } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) pb[q] = mul_rn_range(a.ca, bits_of(x[q]), far);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[q] = __dadd_rn(double_of(pb[q]), y[q]);
            const uint64_t wb = opaque_bits(w[q]);
            bool slow = false;
            uint64_t tb = KIND == 0 ? sqr_rn_core(wb, slow) : mul_rn_quick2(wb, bits_of(z[q]), slow);
            if (slow) {
                tb = mul_hw_bits(wb, KIND == 0 ? wb : bits_of(z[q]));
                left = true;
            }
            t[q] = double_of(tb);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
            element<KIND, MODE>(a, x[q], y[q], KIND == 1 ? z[q] : 0.0, w[q], t[q], left);
    }
}

// Coherent evict-first 32-byte accesses: w may be one of the inputs.
__device__ __forceinline__ void ld4(const double *p, double (&v)[4]) {
    asm volatile("ld.global.cs.v4.f64 {%0,%1,%2,%3}, [%4];"
                 : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3])
                 : "l"(p));
}

__device__ __forceinline__ void st4(double *p, const double (&v)[4]) {
    asm volatile("st.global.cs.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]),
                 "d"(v[2]), "d"(v[3])
                 : "memory");
}

// Terms of the four elements base .. base + 3; w stored.  VEC: one 32-byte
// co-aligned vector of every operand; else element by element with bounds,
// +0 terms past n.
template <int KIND, int MODE, bool VEC, bool EARLY = false>
__device__ __forceinline__ void vector_terms(const ReduceArgs &a, int64_t base, double (&t)[4],
                                             bool &left) {
    if constexpr (VEC) {
        double x[4], y[4], z[4], w[4];
        ld4(a.x + base, x);
        ld4(a.y + base, y);
        if constexpr (KIND == 1) ld4(a.z + base, z);
        elements4<KIND, MODE, EARLY>(a, x, y, z, w, t, left);
        st4(a.w + base, w);
    } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t i = base + q;
            if (i < a.n) {
                const double zi = KIND == 1 ? a.z[i] : 0.0;
                double wi;
                element<KIND, MODE>(a, a.x[i], a.y[i], zi, wi, t[q], left);
                a.w[i] = wi;
            } else {
                t[q] = 0.0;
            }
        }
    }
}

template <int KIND, bool EMU, bool VEC>
__device__ __forceinline__ void vector_terms(const ReduceArgs &a, int64_t base, double (&t)[4]) {
    bool left;
    vector_terms<KIND, EMU ? kInteger : kFp64, VEC>(a, base, t, left);
}

// Bits 6..0 of a tile's tree, by one warp, from the 128 node values that bits
// 12..7 leave (node[j] at position j of a 128-element column, in shared
// memory); valid in lane 0.  Lane l takes positions l + 32 r, so bits 6 and 5
// are three sums in the lane and every further level is one instruction.
__device__ __forceinline__ double column_sum(const double *node, int lane) {
    double v = __dadd_rn(__dadd_rn(node[lane], node[lane + 64]),
                         __dadd_rn(node[lane + 32], node[lane + 96]));
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1) v = __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, sh));
    return v;
}

// The halving tree over the eight values v[0], v[D], .., v[7 D] (three bits, the
// top one first).
template <int D>
__device__ __forceinline__ double tree8(const double *v) {
    return __dadd_rn(__dadd_rn(__dadd_rn(v[0], v[4 * D]), __dadd_rn(v[2 * D], v[6 * D])),
                     __dadd_rn(__dadd_rn(v[D], v[5 * D]), __dadd_rn(v[3 * D], v[7 * D])));
}

}  // namespace

// The cluster form (reduce_split.cu), for kind 0 (norm2) or 1 (dot); vec: every
// pointer 32-byte aligned.  With one tile it writes the result itself.
cudaError_t launch_reduce_split(int kind, bool vec, const ReduceArgs &a, cudaStream_t s);
// The tree over the tile sums, after any form's kernel (reduce_split.cu).
cudaError_t launch_reduce_final(const ReduceArgs &a, cudaStream_t s);

}  // namespace wx
