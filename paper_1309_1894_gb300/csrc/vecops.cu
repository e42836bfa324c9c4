// vecops.cu -- the sibling vector kernels of VecWXPY in the same library:
// VecAXPBYPCZ, VecMAXPY and VecPointwiseMult as streaming kernels, and VecAXPY
// / VecAYPX as the in-place special cases of wxpy().
//
// Definitions (PETSc's, every product and sum rounded to nearest-even in
// binary64, left to right, no fused multiply-add):
//   axpy:      y = RN(RN(alpha*x) + y)                       = wxpy(alpha, x, y) into y
//   aypx:      y = RN(x + RN(alpha*y)) = RN(RN(alpha*y) + x) = wxpy(alpha, y, x) into y
//   axpby:     y = RN(RN(alpha*x) + RN(beta*y))
//   axpbypcz:  z = RN(RN(RN(alpha*x) + RN(beta*y)) + RN(gamma*z))
//   maxpy:     y = RN(... RN(RN(y + RN(a0*x0)) + RN(a1*x1)) ... + RN(a_{m-1}*x_{m-1}))
//   pmult:     w = RN(x*y)
//
// axpby, axpbypcz and maxpy run as one template, the staged kernel below, with
// pointers at any 8-byte offsets; with sums asked for in the integer pipeline and
// offsets that differ by an odd number of elements they, like pointwise_mult where
// offsets differ modulo 32 bytes, take single elements, and pointwise_mult else
// 32-byte vectors.  Every form has an element's inputs loaded before its output is
// stored, so the output may be exactly one of the inputs.
//
// Pipe balance.  On GB300 the FP64 pipeline issues about two operations per
// clock per SM, and these kernels need more of it than wxpy does: axpbypcz
// has 3 products and 2 sums per element (32 bytes of traffic), maxpy with m
// terms 2m operations per 8(m + 2) bytes.  Both are FP64-bound far below the
// HBM roofline unless part of the arithmetic moves to the integer pipelines
// (fp64_emu.cuh, fp64_mul.cuh).  A product costs about twenty ALU operations
// there and a sum about fifty to seventy-five, so products are the cheaper ones to
// move: a runtime fraction (in sixteenths) of each warp's loop iterations
// computes all of its products in the integer pipeline, the rest in FP64;
// the choice is uniform across the warp (no divergence) and rotates with the
// iteration, so every SM sub-partition sees the same mix.  Sums can move too
// (add offload 1: every other one, 2: all; 0: none, but for one or two per pair of
// elements of a wide maxpy group, see integer_sums).  Every split gives the same bits.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "bulk.cuh"
#include "fp64_mul.cuh"
#include "internal.h"

namespace wx {
namespace {

// Coefficients of one launch: as doubles for the FP64 instructions and split
// once on the host for the integer-pipeline products, whose operands' range
// (`from` in each split, `span` here) is the one that suits all of them.
struct Coefs {
    double d[8];
    MulCoef m[8];
    uint32_t span;
};

// What tells that a thread's elements left the fast path of the integer
// pipelines: the products' distance (mul_rn_range), and the sums' word
// (add_rn_quick).
struct Leave {
    uint32_t far = 0, gap = 0;
    __device__ __forceinline__ bool left(const Coefs &c) const {
        return far >= c.span || (int32_t)gap < 0;
    }
};

template <int NIN>
struct EwArgs {
    const double *in[NIN];
    double *out;
    int64_t n, head, nch;  // nch: 4-element chunks (32-byte path) or elements after `head`
    int pm;                // sixteenths of warp iterations whose products run in the integer pipeline
    unsigned odd;          // staged path: inputs an odd number of elements off the output's 16 bytes
    int64_t drop_tile;     // debug: the producer stops before this tile (-1: never)
    Coefs cf;
};

template <int OFF>
__device__ __forceinline__ double add_sel(double a, double b, int position) {
    if constexpr (OFF == 2) return add_rn_int(a, b);
    else if constexpr (OFF == 1) return (position & 1) ? add_rn_int(a, b) : __dadd_rn(a, b);
    else return __dadd_rn(a, b);
}

__device__ __forceinline__ uint64_t bits_of(double v) { return (uint64_t)__double_as_longlong(v); }
__device__ __forceinline__ double double_of(uint64_t b) { return __longlong_as_double((long long)b); }

// p[j] = RN(c_j * e[F + j]), j < K, F = NIN - K (the data operands follow any
// others).  PM = 1: integer-pipeline products, one out-of-line fallback to the
// hardware instruction for the whole element when any of them leaves the
// fast path.  At n = 2^26 (GB300) products with one range test for all of them
// (mul_rn_range) took axpbypcz from 0.92 to 0.965 of the measured peak and maxpy
// with 4 / 8 terms from 0.87 / 0.74 to 0.89 / 0.755, against the fully checked
// ones; there the sums keep the FP64 pipeline at the rate a plain chain of sums
// reaches.
template <int PM, int K, int NIN>
__device__ __forceinline__ void products(const Coefs &c, const double (&e)[NIN], double (&p)[K]) {
    constexpr int F = NIN - K;
    if constexpr (PM == 0) {
#pragma unroll
        for (int j = 0; j < K; ++j) p[j] = __dmul_rn(c.d[j], e[F + j]);
    } else {
        uint32_t far = 0;
        uint64_t b[K];
#pragma unroll
        for (int j = 0; j < K; ++j) b[j] = mul_rn_range(c.m[j], bits_of(e[F + j]), far);
        if (far >= c.span) {
#pragma unroll
            for (int j = 0; j < K; ++j) b[j] = mul_rn_hw_bits(bits_of(c.d[j]), bits_of(e[F + j]));
        }
#pragma unroll
        for (int j = 0; j < K; ++j) p[j] = double_of(b[j]);
    }
}

// The fast path of the integer-pipeline products alone: p[j] as in
// products<1>; one that left the fast path shows in l.far (its bits are then
// meaningless and the caller recomputes the element).  Two distances and the
// largest so far in one instruction: maxpy with 8 terms, n = 2^24, 251 us against
// 257 with one at a time (GB300).
template <int K, int NIN>
__device__ __forceinline__ void products_fast(const Coefs &c, const double (&e)[NIN], double (&p)[K],
                                              Leave &l) {
    constexpr int F = NIN - K;
#pragma unroll
    for (int j = 0; j < K; j += 2) {
        uint32_t d0 = 0, d1 = 0;
        p[j] = double_of(mul_rn_range(c.m[j], bits_of(e[F + j]), d0));
        if (j + 1 < K) p[j + 1] = double_of(mul_rn_range(c.m[j + 1], bits_of(e[F + j + 1]), d1));
        l.far = __vimax3_u32(d0, d1, l.far);
    }
}

template <int OFF>
struct AxpbyOp {
    static constexpr int kIn = 2;  // x, y
    static constexpr bool kStaged = true, kDefaultSums = OFF == 0;
    template <int PM>
    __device__ __forceinline__ static double apply(const Coefs &c, const double (&e)[kIn]) {
        double p[2];
        products<PM>(c, e, p);
        return add_sel<OFF>(p[0], p[1], 1);
    }
    __device__ __forceinline__ static double apply_fast(const Coefs &c, const double (&e)[kIn], int,
                                                        Leave &l) {
        double p[2];
        products_fast(c, e, p, l);
        return add_sel<OFF>(p[0], p[1], 1);
    }
};

template <int OFF>
struct AxpbypczOp {
    static constexpr int kIn = 3;  // x, y, z
    static constexpr bool kStaged = true, kDefaultSums = OFF == 0;
    template <int PM>
    __device__ __forceinline__ static double apply(const Coefs &c, const double (&e)[kIn]) {
        double p[3];
        products<PM>(c, e, p);
        const double s1 = add_sel<OFF>(p[0], p[1], 1);
        return add_sel<OFF>(s1, p[2], OFF == 1 ? 0 : 1);
    }
    __device__ __forceinline__ static double apply_fast(const Coefs &c, const double (&e)[kIn], int,
                                                        Leave &l) {
        double p[3];
        products_fast(c, e, p, l);
        const double s1 = add_sel<OFF>(p[0], p[1], 1);
        return add_sel<OFF>(s1, p[2], OFF == 1 ? 0 : 1);
    }
};

// Which of a maxpy group's sums (bit j: the one that adds term j) run in the
// integer pipeline on the staged kernel's fast path, for the two elements of a
// pair.  The FP64 pipeline does 1.7 sums per clock and SM whatever the code
// (5.0e11/s), so m sums per 8(m + 2) bytes hold these kernels to 0.92 of the HBM
// peak with 4 terms and 0.76 with 8; an integer sum is about 50 ALU operations,
// and there is ALU time left for one or two per pair of elements.  n = 2^24 (GB300), us
// with none / these: 4 terms 137 / 133, 5 169 / 158, 6 204 / 191, 7 237 / 221,
// 8 269 / 246; with 3 terms one of six is slower.  Which of them matters, by
// where it falls among the other sums: 8 terms with sums 0 and 0 264, 3 and 3
// 252.
template <int M>
__device__ constexpr unsigned integer_sums(int q) {
    constexpr unsigned k[7][2] = {{0, 0}, {0, 0}, {1u << 1, 0}, {1u << 2, 0},
                                  {0, 1u << 3}, {0, 1u << 3}, {1u << 2, 1u << 5}};
    return k[M - 2][q];
}

template <int M, int OFF>
struct MaxpyOp {
    static constexpr int kIn = M + 1;  // y, x0 .. x_{M-1}
    static constexpr bool kStaged = true, kDefaultSums = OFF == 0;
    template <int PM>
    __device__ __forceinline__ static double apply(const Coefs &c, const double (&e)[kIn]) {
        double p[M];
        products<PM>(c, e, p);
        double acc = e[0];
#pragma unroll
        for (int j = 0; j < M; ++j) acc = add_sel<OFF>(acc, p[j], j + 1);
        return acc;
    }
    __device__ __forceinline__ static double apply_fast(const Coefs &c, const double (&e)[kIn], int q,
                                                        Leave &l) {
        double p[M];
        products_fast(c, e, p, l);
        double acc = e[0];
#pragma unroll
        for (int j = 0; j < M; ++j) {
            if (OFF == 0 && (integer_sums<M>(q) >> j & 1u))
                acc = double_of(add_rn_quick(j ? opaque_bits(acc) : bits_of(acc), bits_of(p[j]), l.gap));
            else
                acc = add_sel<OFF>(acc, p[j], j + 1);
        }
        return acc;
    }
};

struct PmultOp {
    static constexpr int kIn = 2;
    static constexpr bool kStaged = false, kDefaultSums = false;
    template <int PM>
    __device__ __forceinline__ static double apply(const Coefs &, const double (&e)[kIn]) {
        if constexpr (PM == 1) return double_of(mul_rn_bits(bits_of(e[0]), bits_of(e[1])));
        else return __dmul_rn(e[0], e[1]);
    }
};

template <class Op>
__device__ __forceinline__ void ew_scalar(const EwArgs<Op::kIn> &a, int64_t i) {
    double e[Op::kIn];
#pragma unroll
    for (int k = 0; k < Op::kIn; ++k) {
        double v[1];
        ld_vec<1, 2>(a.in[k] + i, v);
        e[k] = v[0];
    }
    const double r[1] = {Op::template apply<0>(a.cf, e)};
    st_vec<1, 2>(a.out + i, r);
}

// ---- element path: pointers not sharing their offset modulo 32 bytes --------

template <class Op, int PM>
__device__ __forceinline__ void elem_iter(const EwArgs<Op::kIn> &a, int64_t i0, int64_t tpb) {
    constexpr int NIN = Op::kIn, U = NIN <= 3 ? 4 : (NIN <= 5 ? 2 : 1);
    double v[U][NIN];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t i = i0 + u * tpb;
        if (i < a.n) {
#pragma unroll
            for (int k = 0; k < NIN; ++k) {
                double t[1];
                ld_vec<1, 2>(a.in[k] + i, t);
                v[u][k] = t[0];
            }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t i = i0 + u * tpb;
        if (i < a.n) {
            const double r[1] = {Op::template apply<PM>(a.cf, v[u])};
            st_vec<1, 2>(a.out + i, r);
        }
    }
}

template <class Op>
__global__ void __launch_bounds__(256) ew_elem_kernel(const EwArgs<Op::kIn> a) {
    constexpr int U = Op::kIn <= 3 ? 4 : (Op::kIn <= 5 ? 2 : 1);  // as elem_iter
    pdl_enter();
    const int64_t tpb = blockDim.x;
    const int64_t stride = (int64_t)gridDim.x * tpb * U;
    // Warp-uniform rotation through 16 slots; slots below a.pm take the
    // integer-pipeline products.
    unsigned slot = ((threadIdx.x >> 5) * 5u + blockIdx.x * 3u) & 15u;
    for (int64_t i0 = (int64_t)blockIdx.x * tpb * U + threadIdx.x; i0 < a.n; i0 += stride) {
        if ((int)slot < a.pm) elem_iter<Op, 1>(a, i0, tpb);
        else elem_iter<Op, 0>(a, i0, tpb);
        slot = (slot + 1u) & 15u;
    }
}

// ---- direct path: 32-byte register loads, for operations light on arithmetic
// (pointwise_mult: one product per 24 bytes), where a shared-memory ring only
// adds hand-off latency.

template <class Op, int PM>
__device__ __forceinline__ void direct_iter(const EwArgs<Op::kIn> &a, int64_t c0, int64_t tpb) {
    constexpr int NIN = Op::kIn, U = 2;
    double v[U][NIN][4];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t c = c0 + u * tpb;
        if (c < a.nch) {
#pragma unroll
            for (int k = 0; k < NIN; ++k) ld_vec<4, 2>(a.in[k] + a.head + c * 4, v[u][k]);
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int64_t c = c0 + u * tpb;
        if (c < a.nch) {
            double r[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                double e[NIN];
#pragma unroll
                for (int k = 0; k < NIN; ++k) e[k] = v[u][k][q];
                r[q] = Op::template apply<PM>(a.cf, e);
            }
            st_vec<4, 2>(a.out + a.head + c * 4, r);
        }
    }
}

template <class Op>
__global__ void __launch_bounds__(256) ew_direct_kernel(const EwArgs<Op::kIn> a) {
    pdl_enter();
    const int64_t tpb = blockDim.x;
    const int64_t stride = (int64_t)gridDim.x * tpb * 2;
    unsigned slot = ((threadIdx.x >> 5) * 5u + blockIdx.x * 3u) & 15u;
    for (int64_t c0 = (int64_t)blockIdx.x * tpb * 2 + threadIdx.x; c0 < a.nch; c0 += stride) {
        if ((int)slot < a.pm) direct_iter<Op, 1>(a, c0, tpb);
        else direct_iter<Op, 0>(a, c0, tpb);
        slot = (slot + 1u) & 15u;
    }
    // head and tail by the last block (one of its own in a short call)
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 8) {
        const int t = threadIdx.x;
        const int64_t body_end = a.head + a.nch * 4;
        if (t < 4 && t < a.head) ew_scalar<Op>(a, t);
        if (t >= 4 && body_end + (t - 4) < a.n) ew_scalar<Op>(a, body_end + (t - 4));
    }
}

// ---- staged path: bulk copies into a shared-memory ring ----------------------
//
// Eight consumer warps and one producer warp per block; the grid is persistent
// (tiles blockIdx.x, blockIdx.x + gridDim.x, ...).  A tile is TE = 256 * EPT
// elements of every input; the ring holds S tiles.  The producer's lane 0
// waits until all eight consumer warps have released a stage ("empty"
// barrier, one arrival per warp), then issues one bulk copy per input into it
// ("full" barrier, completed by the copies' bytes).  A consumer thread takes
// element pairs 2c, 2c + 512, ... of the tile from shared memory, computes
// them in registers and writes them straight to global memory (16-byte
// stores, coalesced per warp).  Loads never wait on compute: up to S - 1
// tiles are in flight while one is computed, and no register holds a loaded
// vector before its turn.  Each warp picks its product pipe per tile by the
// rotation of ew_elem_kernel; a warp that is ahead runs into the next stage
// without waiting for the others.  Output aliasing: a tile's inputs are in
// shared memory before any of its outputs is written, and no other tile
// touches its addresses, so the output may be one of the inputs.

constexpr int kConsumerWarps = 8;
constexpr int kStagedThreads = 32 * (kConsumerWarps + 1);

// Bitmask of the waits that ran out in this device's kernels (1: producer,
// 2: consumer); read and cleared by wxpy_vecops_status().
__device__ unsigned int g_vec_fault;

// EPT: elements per consumer thread per tile.  MIXED: inputs whose offset from
// the output is odd in elements (see staged_pair), with room for the element
// before and after a tile.
template <int NIN, int EPT, bool MIXED>
struct StageShape {
    static constexpr int kTile = 256 * EPT;
    static constexpr int kStride = kTile + (MIXED ? 2 : 0);  // of an input in a stage
    static constexpr int kTileBytes = NIN * kStride * 8;
    static constexpr int kStages = std::max(2, std::min(4, (72 * 1024) / kTileBytes));
    static constexpr int kSmem = kStages * kTileBytes;
    // three resident blocks for the widest maxpy groups (a register cap of 75
    // measured 6 % faster there; narrower operations gain nothing from it)
    static constexpr int kMinBlocks = NIN >= 7 ? 3 : 2;
};

// The usual tile; calls whose tiles of this length would not give every SM one
// take half of it where there is the choice (65536 elements, GB300: axpbypcz
// 2.25 -> 1.84 us, axpby 1.94 -> 1.69; 262144 and more gain nothing).
template <int NIN>
constexpr int kEpt = NIN <= 3 ? 4 : 2;

__device__ __forceinline__ void ld_shared_v2(const double *p, double &a, double &b) {
    asm volatile("ld.shared.v2.f64 {%0,%1}, [%2];" : "=d"(a), "=d"(b) : "r"(smem_addr(p)));
}

__device__ __forceinline__ void st_global_v2_cs(double *p, double a, double b) {
    asm volatile("st.global.cs.v2.f64 [%0], {%1,%2};" ::"l"(p), "d"(a), "d"(b) : "memory");
}

__device__ __forceinline__ double ld_shared_1(const double *p) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(smem_addr(p)));
    return v;
}

// The j-th two elements of consumer thread c in a tile of `len`: elements 2c + 512 j
// and the next one, in 16-byte accesses; or, MIXED, elements c + 512 j and 256
// further, in single ones.  A bulk copy must start on a 16-byte boundary, so an
// input whose offset from the output is an odd number of elements is copied from
// one element earlier (bit k of `odd`), and its 16-byte pairs would straddle the
// output's; single accesses, 256 contiguous bytes a warp, are free of bank
// conflicts at either offset.  The second element is there if the first is, but
// for MIXED where it says so.
template <class Op, int PM, int EPT, bool MIXED>
__device__ __forceinline__ void staged_pair(const Coefs &cf, const double *sb, double *out, int len,
                                            int c, int j, unsigned odd, Leave &l) {
    constexpr int NIN = Op::kIn;
    using SS = StageShape<NIN, EPT, MIXED>;
    const int p = (MIXED ? c : 2 * c) + 512 * j;
    if (p >= len) return;
    double v[NIN][2];
#pragma unroll
    for (int k = 0; k < NIN; ++k) {
        if constexpr (MIXED) {
            const double *in = sb + k * SS::kStride + (odd >> k & 1u) + p;
            v[k][0] = ld_shared_1(in);
            v[k][1] = p + 256 < len ? ld_shared_1(in + 256) : 1.0;
        } else {
            ld_shared_v2(sb + k * SS::kStride + p, v[k][0], v[k][1]);
        }
    }
    double r[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        double e[NIN];
#pragma unroll
        for (int k = 0; k < NIN; ++k) e[k] = v[k][q];
        if constexpr (PM == 1) r[q] = Op::apply_fast(cf, e, q, l);
        else r[q] = Op::template apply<0>(cf, e);
    }
    if constexpr (MIXED) {
        const double r0[1] = {r[0]}, r1[1] = {r[1]};
        st_vec<1, 2>(out + p, r0);
        if (p + 256 < len) st_vec<1, 2>(out + p + 256, r1);
    } else {
        st_global_v2_cs(out + p, r[0], r[1]);
    }
}

// This thread's elements of a tile, every product in FP64 (PM 0), from the
// stage, which is still held; d: the launch's coefficients.  Out of line: it
// runs only when an integer-pipeline product left its fast path, and inlined
// it would be issued, predicated off, on the FP64 pipeline for every tile.
template <class Op, int EPT, bool MIXED>
__device__ __noinline__ void staged_tile_fp64(double d0, double d1, double d2, double d3,
                                              double d4, double d5, double d6, double d7,
                                              const double *sb, double *out, int len, int c,
                                              unsigned odd) {
    Coefs cf;  // the FP64 products read only the doubles
    cf.d[0] = d0, cf.d[1] = d1, cf.d[2] = d2, cf.d[3] = d3;
    cf.d[4] = d4, cf.d[5] = d5, cf.d[6] = d6, cf.d[7] = d7;
    Leave none;
    for (int j = 0; j < EPT / 2; ++j)
        staged_pair<Op, 0, EPT, MIXED>(cf, sb, out, len, c, j, odd, none);
}

// PM = 1: the integer-pipeline products take their fast path with no test
// between them and the sums, so the tile's arithmetic is one straight run
// that the compiler can interleave (one element's FP64 sums with another's
// integer products); if any product left the fast path, the thread's
// elements are recomputed in FP64 and written again (nothing reads them
// before the kernel ends, and the stage still holds the inputs).  Returns
// whether that happened.
template <class Op, int PM, int EPT, bool MIXED>
__device__ __forceinline__ bool staged_tile(const Coefs &cf, const double *sb, double *out, int len,
                                            int c, unsigned odd) {
    Leave l;
#pragma unroll
    for (int j = 0; j < EPT / 2; ++j)
        staged_pair<Op, PM, EPT, MIXED>(cf, sb, out, len, c, j, odd, l);
    bool left = false;
    if constexpr (PM == 1) {
        left = l.left(cf);
        if (left)
            staged_tile_fp64<Op, EPT, MIXED>(cf.d[0], cf.d[1], cf.d[2], cf.d[3], cf.d[4], cf.d[5],
                                             cf.d[6], cf.d[7], sb, out, len, c, odd);
    }
    return left;
}

template <class Op, int EPT, bool MIXED>
__global__ void __launch_bounds__(kStagedThreads, (StageShape<Op::kIn, EPT, MIXED>::kMinBlocks))
    ew_staged_kernel(const EwArgs<Op::kIn> a) {
    constexpr int NIN = Op::kIn;
    using SS = StageShape<NIN, EPT, MIXED>;
    constexpr int TE = SS::kTile, S = SS::kStages;
    extern __shared__ __align__(128) double ring[];  // [S][NIN][SS::kStride]
    __shared__ __align__(8) uint64_t full[S], empty[S];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t body = a.nch * 4;  // elements from a.head, a multiple of 4
    const int64_t ntiles = (body + TE - 1) / TE;
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(smem_addr(&full[s]), 1);
            mbar_init(smem_addr(&empty[s]), kConsumerWarps);
        }
        mbar_init_fence();
    }
    // The block's first tile on its way into the L2 while the launch before
    // this one ends (a prefetch changes no value), then wait for that launch.
    {
        const int64_t e0 = (int64_t)blockIdx.x * TE;
        const int64_t left = body - e0 < TE ? body - e0 : TE;
        for (int64_t e = 16 * threadIdx.x; e < left; e += 16 * kStagedThreads) {
#pragma unroll
            for (int k = 0; k < NIN; ++k)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(a.in[k] + a.head + e0 + e));
        }
    }
    pdl_wait();
    __syncthreads();
    if (warp == kConsumerWarps) {
        if (lane == 0) {
            const uint64_t policy = evict_first_policy();
            bool ok = true;
            int i = 0;
            for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
                if (t == a.drop_tile) break;
                const int s = i % S;
                if (i >= S && !mbar_wait(smem_addr(&empty[s]), ((i / S) - 1) & 1)) {
                    ok = false;
                    break;
                }
                const int64_t e0 = t * TE;
                const uint32_t len = (uint32_t)(body - e0 < TE ? body - e0 : TE);
                const uint32_t bar = smem_addr(&full[s]);
                mbar_arrive_expect_tx(bar, len * 8u * NIN + (MIXED ? 16u * __popc(a.odd) : 0u));
#pragma unroll
                for (int k = 0; k < NIN; ++k) {
                    const unsigned o = MIXED ? a.odd >> k & 1u : 0u;
                    bulk_load(smem_addr(ring + ((size_t)s * NIN + k) * SS::kStride),
                              a.in[k] + a.head + e0 - o, (len + 2u * o) * 8u, bar, policy);
                }
            }
            // Every issued copy lands before the block exits (the earlier
            // ones were consumed before their stage was reused).
            for (int j = i > S ? i - S : 0; j < i; ++j)
                if (!mbar_wait(smem_addr(&full[j % S]), (j / S) & 1)) ok = false;
            if (!ok) atomicOr(&g_vec_fault, 1u);
        }
    } else {
        // Head and tail elements (four each at most) by eight lanes of the last
        // block, while its first tile is on its way: at the end they were a
        // memory latency of their own (65536 elements, 8 bytes off, GB300:
        // axpbypcz 2.7 us, 1.95 here).
        if (blockIdx.x == gridDim.x - 1 && warp == kConsumerWarps - 1 && lane < 8) {
            const int64_t e = lane < 4 ? lane : a.head + body + (lane - 4);
            if (lane < 4 ? e < a.head : e < a.n) ew_scalar<Op>(a, e);
        }
        unsigned slot = (warp * 5u + blockIdx.x * 3u) & 15u;
        int i = 0, fp64 = 0;
        for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x, ++i) {
            const int s = i % S;
            if (!mbar_wait(smem_addr(&full[s]), (i / S) & 1)) {
                if (lane == 0) atomicOr(&g_vec_fault, 2u);
                break;
            }
            const int64_t e0 = t * TE;
            const int len = (int)(body - e0 < TE ? body - e0 : TE);
            const double *sb = ring + (size_t)s * NIN * SS::kStride;
            double *out = a.out + a.head + e0;
            // Data that keeps leaving the fast path (zeros, say) pays for both
            // kinds of product: after a tile where a quarter of the lanes did,
            // the warp takes FP64 products for sixteen tiles.  Every seventh
            // element zero, maxpy with 4 terms, n = 2^26 (GB300): 1065 us
            // against 1557.
            bool left = false;
            if ((int)slot < a.pm && fp64 == 0)
                left = staged_tile<Op, 1, EPT, MIXED>(a.cf, sb, out, len, threadIdx.x, a.odd);
            else staged_tile<Op, 0, EPT, MIXED>(a.cf, sb, out, len, threadIdx.x, a.odd);
            fp64 = __popc(__ballot_sync(0xffffffffu, left)) > 8 ? 16 : fp64 > 0 ? fp64 - 1 : 0;
            mbar_arrive_warp(smem_addr(&empty[s]), lane);
            slot = (slot + 1u) & 15u;
        }
        // The next launch may start now, not before: blocks that come while these
        // compute take what room there is, unevenly, and it is the fullest SM
        // that ends the grid (262144 elements back to back, axpbypcz 4.4 us when
        // they come at the start, 3.45 here; maxpy with 8 terms on 131075, 5.7
        // and 4.9).
        pdl_trigger();
    }
}

// Per device: the dynamic shared-memory opt-in done and the resident blocks
// per SM of one staged kernel.
template <class Op, int EPT, bool MIXED>
int staged_blocks_per_sm(int device) {
    static std::atomic<int> cached[64];
    if (device < 0 || device >= 64) return 0;
    int v = cached[device].load(std::memory_order_relaxed);
    if (v > 0) return v;
    constexpr int smem = StageShape<Op::kIn, EPT, MIXED>::kSmem;
    if (cudaFuncSetAttribute(ew_staged_kernel<Op, EPT, MIXED>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return 0;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, ew_staged_kernel<Op, EPT, MIXED>,
                                                      kStagedThreads, smem) != cudaSuccess || nb < 1)
        return 0;
    cached[device].store(nb, std::memory_order_relaxed);
    return nb;
}

template <class Op, int EPT, bool MIXED>
cudaError_t launch_staged(const EwArgs<Op::kIn> &a, const DeviceProps *dp, cudaStream_t s) {
    using SS = StageShape<Op::kIn, EPT, MIXED>;
    const int nb = staged_blocks_per_sm<Op, EPT, MIXED>(dp->device);
    if (nb == 0) {
        const cudaError_t e = cudaGetLastError();
        return e == cudaSuccess ? cudaErrorInvalidConfiguration : e;
    }
    const int64_t tiles = (a.nch * 4 + SS::kTile - 1) / SS::kTile;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((int64_t)dp->sm_count * nb, tiles));
    return launch_pdl_smem(&ew_staged_kernel<Op, EPT, MIXED>, (unsigned)grid, kStagedThreads,
                           SS::kSmem, s, a);
}

std::atomic<long long> g_drop_tile{-1};

// Validation shared by the three streaming operations: n >= 0, 8-byte aligned
// non-null pointers, and the output either disjoint from or exactly equal to
// each input.
int validate(int64_t n, const double *const *in, int nin, const double *out) {
    if (n < 0) return fail(WXPY_EINVAL, "n = %lld is negative", (long long)n);
    if (n == 0) return WXPY_OK;
    if (n > ((int64_t)1 << 56)) return fail(WXPY_EINVAL, "n too large");
    const uint64_t bytes = (uint64_t)n * 8;
    const uintptr_t po = (uintptr_t)out;
    if (!out || (po & 7)) return fail(WXPY_EINVAL, "null or misaligned output");
    for (int k = 0; k < nin; ++k) {
        const uintptr_t p = (uintptr_t)in[k];
        if (!in[k] || (p & 7)) return fail(WXPY_EINVAL, "null or misaligned input %d", k);
        if (p != po && p < po + bytes && po < p + bytes)
            return fail(WXPY_EOVERLAP, "output partially overlaps input %d", k);
    }
    return WXPY_OK;
}

template <class Op>
int launch_ew(const double *const *in, double *out, int64_t n, const double *coef, int ncoef,
              int pm, cudaStream_t s) {
    constexpr int NIN = Op::kIn;
    int st = validate(n, in, NIN, out);
    if (st != WXPY_OK || n == 0) return st;
    const DeviceProps *dp = current_device(&st);
    if (!dp) return st;
    EwArgs<NIN> a;
    uintptr_t diff = 0;
    for (int k = 0; k < NIN; ++k) {
        a.in[k] = in[k];
        diff |= (uintptr_t)in[k] ^ (uintptr_t)out;
    }
    a.out = out;
    a.n = n;
    a.pm = pm;
    a.drop_tile = g_drop_tile.load();
    uint32_t from = 0, to = ~0u;
    for (int k = 0; k < 8; ++k) {
        a.cf.d[k] = k < ncoef ? coef[k] : 0.0;
        uint64_t b;
        std::memcpy(&b, &a.cf.d[k], 8);
        a.cf.m[k] = mul_coef_of(b);
        if (k < ncoef) {
            from = std::max(from, a.cf.m[k].from);
            to = std::min(to, a.cf.m[k].from + a.cf.m[k].span);
        }
    }
    // coefficients that share no range (one of them zero, say): FP64 products
    a.cf.span = to > from ? to - from : 0u;
    if (ncoef > 0 && a.cf.span == 0) a.pm = 0;
    for (MulCoef &m : a.cf.m) m.from = from;
    cudaError_t e = injected_launch_error();
    if (e != cudaSuccess) return fail_cuda(e, "vector kernel launch");
    a.odd = 0;
    for (int k = 0; k < NIN; ++k)
        if (((uintptr_t)in[k] ^ (uintptr_t)out) & 8u) a.odd |= 1u << k;
    // The staged body wants its inputs at the output's place in 16 bytes, the
    // direct one in 32; with the default sums the staged one takes any offset.
    // Single elements from registers, the path they replace, ran axpbypcz and
    // maxpy with 5 / 8 terms at 0.81 and 0.78 / 0.68 of the measured peak with
    // differing offsets (n = 2^26, GB300), against 0.97 and 0.81 / 0.76 staged.
    if (Op::kStaged ? a.odd == 0 || Op::kDefaultSums : (diff & 31u) == 0) {
        // peel the head to the output's 32-byte boundary
        a.head = std::min<int64_t>((4 - (int64_t)(((uintptr_t)out >> 3) & 3)) & 3, n);
        a.nch = (n - a.head) / 4;
        if (a.odd) {
            // the copies reach one element before the body and one past it
            if (a.head == 0) a.head = std::min<int64_t>(4, n);
            a.nch = std::max<int64_t>(0, n - a.head - 1) / 4;
        }
        if constexpr (Op::kStaged) {
            constexpr int EPT = kEpt<NIN>;
            if constexpr (Op::kDefaultSums) {
                const bool small = EPT > 2 && a.nch * 4 < (int64_t)dp->sm_count * 256 * EPT;
                if (a.odd) e = small ? launch_staged<Op, 2, true>(a, dp, s) : launch_staged<Op, EPT, true>(a, dp, s);
                else e = small ? launch_staged<Op, 2, false>(a, dp, s) : launch_staged<Op, EPT, false>(a, dp, s);
            } else {
                e = launch_staged<Op, EPT, false>(a, dp, s);
            }
        } else {
            const int64_t per_block = 256 * 2;
            const int64_t edges = a.head + 4 * a.nch != a.n || a.head != 0;
            const int64_t grid = std::max<int64_t>(
                1, std::min<int64_t>((int64_t)dp->sm_count * 8,
                                     (a.nch + per_block - 1) / per_block + edges));
            e = launch_pdl(&ew_direct_kernel<Op>, (unsigned)grid, 256, s, a);
        }
    } else {
        a.head = 0;
        a.nch = n;
        const int64_t per_block = 256 * 4;
        const int64_t grid = std::max<int64_t>(
            1, std::min<int64_t>((int64_t)dp->sm_count * 8, (n + per_block - 1) / per_block));
        e = launch_pdl(&ew_elem_kernel<Op>, (unsigned)grid, 256, s, a);
    }
    if (e != cudaSuccess) return fail_cuda(e, "vector kernel launch");
    return WXPY_OK;
}

// Pipe split: add offload (0, 1, 2) and product sixteenths (0..16); -1 in
// either leaves the operation's searched split, else its default (below).
std::atomic<int> g_vec_add{-1};
std::atomic<int> g_vec_mul{-1};
std::atomic<int> g_vec_tuned[2][WXPY_VEC_CLASSES] = {{-1, -1, -1, -1, -1, -1, -1, -1, -1, -1},
                                                     {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1}};
std::atomic<int> g_vec_last[WXPY_VEC_CLASSES];  // the range stored last

constexpr int64_t kLongCall = (int64_t)1 << 23;  // elements: HBM's side of vecops_default

using Pipes = VecPipes;

Pipes pipes_for(int cls, int64_t n) {
    Pipes p = vecops_default(cls, n);
    vecops_tuned_load(cls, vecops_range(n), &p);
    const int add = g_vec_add.load(), mul = g_vec_mul.load();
    if (add >= 0) p.add = add;
    if (mul >= 0) p.mul = mul;
    return p;
}

template <int M>
int maxpy_group(int64_t n, const double *alpha, const double *const *in, Pipes p, cudaStream_t s) {
    switch (p.add) {
        case 0: return launch_ew<MaxpyOp<M, 0>>(in, (double *)in[0], n, alpha, M, p.mul, s);
        case 1: return launch_ew<MaxpyOp<M, 1>>(in, (double *)in[0], n, alpha, M, p.mul, s);
        default: return launch_ew<MaxpyOp<M, 2>>(in, (double *)in[0], n, alpha, M, p.mul, s);
    }
}

}  // namespace

// Defaults, measured on GB300 (the product share that balanced the FP64 and ALU
// pipelines best).  In calls that the L2 serves the fewer FP64 instructions the
// better; where HBM sets the pace a few FP64 products are free and shorter.
// us at 10^6 / 4x10^6 / 2^24 / 2^26 elements: axpby with all products integer
// 4.8 / 14.2 / 68.0 / 263, with 10/16 6.2 / 17.7 / 66.1 / 245; axpbypcz 6.6 /
// 20.1 / 82.5 / 320, 15/16 7.1 / 21.3 / 82.5 / 315; maxpy with two terms 6.6 /
// 19.1 / 84.5 / 332, 14/16 7.3 / 21.6 / 82.1 / 313.
VecPipes vecops_default(int cls, int64_t n) {
    if (cls == WXPY_VEC_PMULT) return {0, 4};
    const bool short_call = vecops_range(n) == 0;
    if (cls == WXPY_VEC_AXPBYPCZ) return {0, short_call ? 16 : 15};
    if (cls == WXPY_VEC_AXPBY) return {0, short_call ? 16 : 10};
    return {0, cls + 1 == 2 && !short_call ? 14 : 16};  // maxpy with cls + 1 terms
}

int vecops_inputs(int cls) {
    if (cls == WXPY_VEC_AXPBYPCZ) return 3;
    if (cls == WXPY_VEC_PMULT || cls == WXPY_VEC_AXPBY) return 2;
    return cls + 2;  // y and cls + 1 x vectors
}

int vecops_range(int64_t n) { return n < kLongCall ? 0 : 1; }

bool vecops_tuned_load(int cls, int range, VecPipes *p) {
    if (cls < 0 || cls >= WXPY_VEC_CLASSES) return false;
    const int v = g_vec_tuned[range < 0 ? g_vec_last[cls].load() : range][cls].load();
    if (v < 0) return false;
    p->add = v >> 5;
    p->mul = v & 31;
    return true;
}

void vecops_tuned_store(int cls, int range, const VecPipes *p) {
    if (cls < 0 || cls >= WXPY_VEC_CLASSES) return;
    for (int r = 0; r < 2; ++r)
        if (range < 0 || range == r) {
            g_vec_tuned[r][cls].store(p ? (p->add << 5) | p->mul : -1);
            g_vec_last[cls].store(r);
        }
}

int vecops_run(int cls, int64_t n, const double *coef, const double *const *in, double *out,
               VecPipes p, cudaStream_t s) {
    switch (cls) {
        case WXPY_VEC_AXPBYPCZ:
            switch (p.add) {
                case 0: return launch_ew<AxpbypczOp<0>>(in, out, n, coef, 3, p.mul, s);
                case 1: return launch_ew<AxpbypczOp<1>>(in, out, n, coef, 3, p.mul, s);
                default: return launch_ew<AxpbypczOp<2>>(in, out, n, coef, 3, p.mul, s);
            }
        case WXPY_VEC_PMULT: return launch_ew<PmultOp>(in, out, n, nullptr, 0, p.mul, s);
        case WXPY_VEC_AXPBY:
            switch (p.add) {
                case 0: return launch_ew<AxpbyOp<0>>(in, out, n, coef, 2, p.mul, s);
                default: return launch_ew<AxpbyOp<2>>(in, out, n, coef, 2, p.mul, s);
            }
        case 1: return maxpy_group<2>(n, coef, in, p, s);
        case 2: return maxpy_group<3>(n, coef, in, p, s);
        case 3: return maxpy_group<4>(n, coef, in, p, s);
        case 4: return maxpy_group<5>(n, coef, in, p, s);
        case 5: return maxpy_group<6>(n, coef, in, p, s);
        case 6: return maxpy_group<7>(n, coef, in, p, s);
        case 7: return maxpy_group<8>(n, coef, in, p, s);
        default: return fail(WXPY_EINVAL, "bad vector kernel class %d", cls);
    }
}

}  // namespace wx

using namespace wx;

extern "C" {

int wxpy_axpy(int64_t n, double alpha, const double *x, double *y, void *stream) {
    return wxpy(n, alpha, x, y, y, stream);
}

int wxpy_aypx(int64_t n, double alpha, const double *x, double *y, void *stream) {
    return wxpy(n, alpha, y, x, y, stream);
}

int wxpy_axpby(int64_t n, double alpha, double beta, const double *x, double *y, void *stream) {
    const double *in[2] = {x, y};
    const double coef[2] = {alpha, beta};
    return vecops_run(WXPY_VEC_AXPBY, n, coef, in, y, pipes_for(WXPY_VEC_AXPBY, n),
                      (cudaStream_t)stream);
}

int wxpy_axpbypcz(int64_t n, double alpha, double beta, double gamma, const double *x,
                  const double *y, double *z, void *stream) {
    const double *in[3] = {x, y, z};
    const double coef[3] = {alpha, beta, gamma};
    return vecops_run(WXPY_VEC_AXPBYPCZ, n, coef, in, z, pipes_for(WXPY_VEC_AXPBYPCZ, n),
                      (cudaStream_t)stream);
}

int wxpy_maxpy(int64_t n, int m, const double *alpha, const double *const *x, double *y,
               void *stream) {
    if (m < 0) return fail(WXPY_EINVAL, "negative m");
    if (m > 0 && (!alpha || !x)) return fail(WXPY_EINVAL, "null alpha or x array");
    if (m == 0 || n == 0) {
        const double *none[1] = {y};
        return validate(n, none, 1, y);
    }
    cudaStream_t s = (cudaStream_t)stream;
    // Groups of at most 8 terms, in order: y itself carries the rounded
    // partial sum from one group to the next, as the definition requires.
    for (int j0 = 0; j0 < m; j0 += 8) {
        const int g = std::min(8, m - j0);
        int st;
        if (g == 1) {
            // a single term is y = RN(y + RN(a x)) = RN(RN(a x) + y): wxpy into y
            st = wxpy(n, alpha[j0], x[j0], y, y, stream);
        } else {
            const double *in[9];
            in[0] = y;
            for (int j = 0; j < g; ++j) in[j + 1] = x[j0 + j];
            st = vecops_run(g - 1, n, alpha + j0, in, y, pipes_for(g - 1, n), s);
        }
        if (st != WXPY_OK) return st;
    }
    return WXPY_OK;
}

int wxpy_pointwise_mult(int64_t n, const double *x, const double *y, double *w, void *stream) {
    const double *in[2] = {x, y};
    return vecops_run(WXPY_VEC_PMULT, n, nullptr, in, w, pipes_for(WXPY_VEC_PMULT, n),
                      (cudaStream_t)stream);
}

int wxpy_vecops_pipes(int add_offload, int mul_sixteenths) {
    if (add_offload < -1 || add_offload > 2)
        return fail(WXPY_EINVAL, "add offload must be -1, 0, 1 or 2");
    if (mul_sixteenths < -1 || mul_sixteenths > 16)
        return fail(WXPY_EINVAL, "product sixteenths must be in -1..16");
    g_vec_add.store(add_offload);
    g_vec_mul.store(mul_sixteenths);
    return WXPY_OK;
}

int wxpy_vecops_status(void) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    unsigned int fault = 0;
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(&fault, g_vec_fault, sizeof(fault));
    const unsigned int zero = 0;
    if (e == cudaSuccess && fault) e = cudaMemcpyToSymbol(g_vec_fault, &zero, sizeof(zero));
    if (e != cudaSuccess) return fail_cuda(e, "vector kernel status");
    if (fault)
        return fail(WXPY_ETIMEOUT, "a staged vector kernel's bounded wait ran out (%s)",
                    fault & 1u ? (fault & 2u ? "producer and consumers" : "producer") : "consumers");
    return WXPY_OK;
}

int wxpy_debug_vecops_split(int op_class, int64_t n, int *add_offload, int *mul_sixteenths) {
    if (op_class < 0 || op_class >= WXPY_VEC_CLASSES || n < 0 || !add_offload || !mul_sixteenths)
        return fail(WXPY_EINVAL, "bad vector class %d or size", op_class);
    const Pipes p = pipes_for(op_class, n);
    *add_offload = p.add;
    *mul_sixteenths = p.mul;
    return WXPY_OK;
}

int wxpy_debug_vecops_drop_tile(int64_t tile) {
    if (tile < -1) return fail(WXPY_EINVAL, "tile must be >= -1");
    g_drop_tile.store(tile);
    return WXPY_OK;
}

}  // extern "C"
