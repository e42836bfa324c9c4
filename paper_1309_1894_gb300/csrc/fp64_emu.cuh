// fp64_emu.cuh -- IEEE 754 binary64 addition, round to nearest even, computed
// in the integer pipeline.
//
// Why.  w = RN(RN(alpha*x) + y) needs two FP64 instructions per element (the
// two roundings forbid a fused multiply-add), and on GB300 the FP64 pipeline
// issues only about two operations per clock per SM: a 256-bit streaming
// kernel doing DMUL+DADD reaches about 6.0 TB/s, the same kernel with one FP64
// instruction per element 7.2 TB/s.  The integer pipeline is nearly idle in
// this kernel, so part or all of the additions are moved there, which lifts the
// FP64 ceiling above the HBM one.
//
// Method (the definition of a correctly rounded sum, on integer significands).
// For two normal operands, order them by magnitude, |hi| >= |lo|.  Place hi's
// 53-bit significand (hidden bit included) at bits 62..10 of a 64-bit integer
// and lo's likewise, then shift lo's right by the exponent difference d; every
// bit shifted out is OR-ed into bit 0 (a "sticky" or jamming bit).  Add the
// two integers when the signs agree (renormalising a carry into bit 63 by one
// right shift, again jamming) or subtract them when they differ (an exact zero
// gives +0; otherwise shift the leading one back to bit 62).  Round at bit 10:
// up if the ten bits below are more than half, to even on exactly half.
// Correctness of the jamming bit: the bits below the rounding point are only
// approximated when bits were shifted out (d > 10); the approximation is then
// the floor or the ceiling of the exact value on a grid ten bits finer than
// the rounding point, with bit 0 set, so it is never the exact-half pattern and
// compares with one half exactly as the exact value does.  A subtraction with
// d >= 2 renormalises by at most one bit, so nine guard bits stay; with d <= 1
// nothing is shifted out and the result is exact before rounding.
// Operands that are zero, subnormal, infinite or NaN, and sums whose rounded
// result would be subnormal or overflow, take the hardware instruction
// (__dadd_rn) instead; for finite data in the normal range that never happens.
#pragma once

#include <cstdint>

#include "fp64_mul.cuh"

// The sum (add_rn_with) also compiles as plain host C++, so the host can
// check it against its own IEEE addition.
#ifdef __CUDACC__
#define WX_EMU_FN __device__ __forceinline__
#else
#define WX_EMU_FN inline
#endif

namespace wx {

// RN(a + b) on the bit patterns ua, ub of two binary64 values.  Operands and
// results the integer path leaves out go to hw(ua, ub): the hardware
// instruction, out of line, in the kernels (add_rn_bits below); the host's
// check of this function passes a recorder instead.
template <class Hw>
WX_EMU_FN uint64_t add_rn_with(uint64_t ua, uint64_t ub, Hw hw) {
    constexpr uint64_t kSign = 1ull << 63;
    constexpr uint64_t kAbs = kSign - 1;
    constexpr uint64_t kFrac = (1ull << 52) - 1;
    constexpr uint64_t kHidden = 1ull << 52;
    const bool a_big = (ua & kAbs) >= (ub & kAbs);
    const uint64_t hi = a_big ? ua : ub;
    const uint64_t lo = a_big ? ub : ua;
    const int ehi = (int)((hi >> 52) & 0x7FF);
    const int elo = (int)((lo >> 52) & 0x7FF);
    // Inf/NaN, zero or subnormal operands go to the hardware at the end.
    bool slow = ehi == 0x7FF || elo == 0;
    // Branch-free from here to the single fallback test: the lanes of a warp
    // follow one path whatever the signs and exponent gaps of their operands.
    // Every value stays an integer bit pattern until the one reinterpretation
    // at the end: merging several double-valued return paths made the
    // compiler issue FP64-pipeline instructions.
#ifdef __CUDA_ARCH__
    const int dd = min(ehi - elo, 63);  // a gap of 63 or more leaves only the sticky bit
#else
    const int dd = ehi - elo < 63 ? ehi - elo : 63;
#endif
    const uint64_t H = ((hi & kFrac) | kHidden) << 10;
    const uint64_t L0 = ((lo & kFrac) | kHidden) << 10;
    const uint64_t L = (L0 >> dd) | (uint64_t)((L0 & ((1ull << dd) - 1)) != 0);
    // H + L, or H - L (two's complement) when the signs differ
    const uint64_t neg = ((hi ^ lo) & kSign) ? ~0ull : 0ull;
    uint64_t S = H + (L ^ neg) - neg;
    const bool zero = S == 0;  // exact cancellation rounds to +0
    // Leading one back to bit 62: one right shift after a carry (lz == 0, with
    // the jam bit kept), or lz - 1 left shifts after a cancellation.
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)S);
#else
    const int lz = S ? __builtin_clzll(S) : 64;
#endif
    const uint64_t right = (S >> 1) | (S & 1);
    const uint64_t left = S << ((lz - 1) & 63);
    S = lz == 0 ? right : left;
    int e = ehi + 1 - lz;
    // Round to nearest, ties to even, at bit 10.
    uint64_t m = S >> 10;
    const uint64_t rem = S & 0x3FF;
    m += (uint64_t)(rem > 0x200 || (rem == 0x200 && (m & 1)));
    const int carry = (int)(m >> 53);  // rounding reached the next binade
    m >>= carry;
    e += carry;
    slow = slow || (!zero && (e <= 0 || e >= 0x7FF));  // subnormal or overflowing result
    uint64_t bits = zero ? 0ull : ((hi & kSign) | ((uint64_t)e << 52) | (m & kFrac));
    if (slow) bits = hw(ua, ub);
    return bits;
}

// RN(a + b) with the cheapest checks, for kernels that move a few of many sums:
// ORs into `away` a word whose top bit is set when the operands leave the fast
// path (the bits are then meaningless): the larger magnitude's exponent field
// outside [64, 2015], or a difference that cancels 20 bits or more.  Every gap
// between the two is taken, and a zero or subnormal smaller one, which is 64 or
// more below and counts as a number of that exponent field.
//
// Method, in 32-bit words.  The larger operand's significand, hidden bit at bit
// 19 of the top word, and the smaller one's shifted right by the gap are held in
// 96 bits; they are added, or subtracted as a two's complement when the signs
// differ.  The shift is made in two parts, by up to 32 bits and by the rest, and
// `lost` is not 0 exactly when bits of it leave the 96 (gaps of 33 and more;
// from 63 on the smaller one counts as about that far below, and no bit of the
// result depends on how far).  A sum with lost bits lies above the 96 bits by
// less than one of them; a difference lies below, so its complement leaves out
// the final one and then lies above as well.  The sum's leading bit is at bit 20
// or below, so one left shift puts it there.  The lowest word is then all that
// is rounded away, and adding one half to it carries into the significand
// exactly when it is at least one half; it becomes 0 with nothing lost exactly
// on a tie, which clears the lowest bit.
WX_EMU_FN uint64_t add_rn_quick(uint64_t ua, uint64_t ub, uint32_t &away) {
    const uint32_t ah = (uint32_t)(ua >> 32), al = (uint32_t)ua;
    const uint32_t bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
    const uint32_t A = ah & 0x7FFFFFFFu, B = bh & 0x7FFFFFFFu;
    const bool b_big = A < B;
    const uint32_t H = b_big ? B : A, L = b_big ? A : B;
    const uint32_t hl = b_big ? bl : al, ll = b_big ? al : bl, hh = b_big ? bh : ah;
    const uint32_t x = H - (L & 0x7FF00000u);  // gap << 20, and fraction bits below
    const uint32_t d = (x + 0x100000u) >> 20;  // gap + 1
    const uint32_t hm = (H & 0xFFFFFu) | 0x100000u, lm = (L & 0xFFFFFu) | 0x100000u;
    const uint32_t m = (uint32_t)((int32_t)(ah ^ bh) >> 31);
    const uint32_t e = d > 32u ? d - 32u : 0u;  // the shift's second part
    const uint32_t r1 = funnel_rc(ll, lm, d), r0 = funnel_rc(0u, ll, d);
    const uint32_t t2 = funnel_rc(lm, 0u, d), t1 = funnel_rc(r1, 0u, e), t0 = funnel_rc(r0, r1, e);
    const uint32_t lost = funnel_rc(0u, r0, e);
    uint32_t s2, s1, s0;
#ifdef __CUDA_ARCH__
    uint32_t drop;
    asm("add.cc.u32 %3, %4, 1;\n\t"  // carry in: 1 to subtract
        "addc.cc.u32 %0, %5, %6;\n\t"
        "addc.cc.u32 %1, %7, %8;\n\t"
        "addc.u32 %2, %9, %10;"
        : "=r"(s0), "=r"(s1), "=r"(s2), "=r"(drop)
        : "r"(m & ~lost), "r"(hl << 31), "r"(t0 ^ m), "r"(funnel_r(hl, hm, 1u)), "r"(t1 ^ m), "r"(hm >> 1),
          "r"(t2 ^ m));
    const int lz = __clz((int)s2);
#else
    const uint64_t w0 = (uint64_t)(hl << 31) + (t0 ^ m) + (lost == 0u ? m & 1u : 0u);
    const uint64_t w1 = (uint64_t)funnel_r(hl, hm, 1u) + (t1 ^ m) + (w0 >> 32);
    s0 = (uint32_t)w0, s1 = (uint32_t)w1, s2 = (hm >> 1) + (t2 ^ m) + (uint32_t)(w1 >> 32);
    const int lz = s2 ? __builtin_clz(s2) : 32;
#endif
    away |= (H - (64u << 20)) | ((2016u << 20) - 1u - H) | (s2 - 1u);
    const uint32_t n = (uint32_t)lz - 11u;  // left shift: leading bit to bit 20
    const uint32_t r = 32u - n;
    // left funnels as right ones of the neighbouring words (n in 0..20)
#ifdef __CUDA_ARCH__
    const uint32_t o2 = __funnelshift_l(s1, s2, n), o1 = __funnelshift_l(s0, s1, n);
    const uint32_t g = s0 << (n & 31u);
    (void)r;
#else
    const uint32_t o2 = n ? (s2 << n) | (uint32_t)((uint64_t)s1 >> (r & 63u)) : s2;
    const uint32_t o1 = n ? (s1 << n) | (uint32_t)((uint64_t)s0 >> (r & 63u)) : s1;
    const uint32_t g = s0 << (n & 31u);
#endif
    const uint32_t hw = (hh & 0xFFF00000u) + (o2 - (n << 20));
    uint32_t gs, lo, hi;
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %3, 0x80000000;\n\t"
        "addc.cc.u32 %1, %4, 0;\n\t"
        "addc.u32 %2, %5, 0;"
        : "=r"(gs), "=r"(lo), "=r"(hi)
        : "r"(g), "r"(o1), "r"(hw));
#else
    gs = g + 0x80000000u;
    lo = o1 + (g >> 31);
    hi = hw + (uint32_t)(lo < o1);
#endif
    lo = (gs | lost) == 0u ? lo & ~1u : lo;
    return ((uint64_t)hi << 32) | lo;
}

#ifdef __CUDACC__

// The hardware sum for the rare operands the integer path leaves out, on bit
// patterns.  Kept out of line: an inlined fallback is if-converted by the
// compiler -- issued, predicated off, for every element -- and would occupy the
// FP64 pipeline the integer path exists to relieve; and its arguments and
// result are integers, since the moves that set up double-typed call
// arguments were issued for every element as well.
static __device__ __noinline__ uint64_t add_rn_hw_bits(uint64_t ua, uint64_t ub) {
    return (uint64_t)__double_as_longlong(
        __dadd_rn(__longlong_as_double((long long)ua), __longlong_as_double((long long)ub)));
}

// The bit pattern of a double through an opaque register move.  Handing the
// integer path a value the compiler still sees as a double (for instance the
// product just computed) let it rewrite integer operations on its bits into
// FP64-pipeline instructions.
__device__ __forceinline__ uint64_t opaque_bits(double v) {
    uint64_t b;
    asm volatile("mov.b64 %0, %1;" : "=l"(b) : "d"(v));
    return b;
}

struct AddRnHw {
    __device__ __forceinline__ uint64_t operator()(uint64_t ua, uint64_t ub) const {
        return add_rn_hw_bits(ua, ub);
    }
};

// RN(a + b) on the bit patterns ua, ub of two binary64 values.
__device__ __forceinline__ uint64_t add_rn_bits(uint64_t ua, uint64_t ub) {
    return add_rn_with(ua, ub, AddRnHw{});
}

__device__ __forceinline__ double add_rn_int(double a, double b) {
    return __longlong_as_double((long long)add_rn_bits(opaque_bits(a), opaque_bits(b)));
}

// w = RN(RN(alpha*x) + y) for VW elements; the sum of element k runs in the
// integer pipeline when EMU == 2, or when EMU == 1 and (base + k) is odd.
template <int VW, int EMU>
__device__ __forceinline__ void wxpy_vec_emu(double alpha, const double (&x)[VW],
                                             const double (&y)[VW], double (&w)[VW], int base) {
    static_assert(EMU >= 0 && EMU <= 2, "the product offload needs the coefficient split");
#pragma unroll
    for (int k = 0; k < VW; ++k) {
        const double p = __dmul_rn(alpha, x[k]);
        const bool emu = EMU == 2 || (EMU == 1 && ((base + k) & 1));
        w[k] = emu ? add_rn_int(p, y[k]) : __dadd_rn(p, y[k]);
    }
}

// How a vector of integer-pipeline products tells operands that it leaves out.
// kTestEach: a test for each product, over its whole range of operands.  A
// product's sum waits for its own x alone, which is what the single-call kernels
// want, whose threads have one or two vectors: 2^20 elements 4.31 us on GB300, 16
// bytes off 4.34, against 4.52 and 5.41 with one test for the vector.
// kTestVector: one test for the vector, over the same range, in the batched
// kernel's wide body: 4096 segments up to 2^18, 316 us, with every seventh element
// zero 383, against 317 and 405.  kTestWindow: one test for the vector and half
// the exponents (mul_rn_quick), in the batched body with three resident blocks,
// which has no register to spare for more.
enum ProductTest { kTestEach, kTestVector, kTestWindow };

// The same with alpha's split `ca` at hand: EMU == 3 computes every product
// RN(alpha*x) in the integer pipelines (fp64_mul.cuh; operands it leaves out take
// the hardware multiply, out of line) and every sum on the FP64 pipeline, which
// then carries one instruction per element.
template <int VW, int EMU, ProductTest TEST = kTestEach>
__device__ __forceinline__ void wxpy_vec_emu(double alpha, const MulCoef &ca, const double (&x)[VW],
                                             const double (&y)[VW], double (&w)[VW], int base) {
    if constexpr (EMU == 3 && TEST == kTestEach) {
#pragma unroll
        for (int k = 0; k < VW; ++k) {
            const uint64_t xb = (uint64_t)__double_as_longlong(x[k]);
            uint32_t far = 0;
            uint64_t p = mul_rn_range(ca, xb, far);
            if (far >= ca.span) p = mul_rn_hw_bits((uint64_t)__double_as_longlong(alpha), xb);
            w[k] = __dadd_rn(__longlong_as_double((long long)p), y[k]);
        }
    } else if constexpr (EMU == 3) {
        static_assert(VW % 2 == 0, "the fallback takes two at a time");
        constexpr bool WINDOW = TEST == kTestWindow;
        uint32_t far = WINDOW && ca.win == 0 ? 1u << 31 : 0u;
        uint64_t p[VW];
#pragma unroll
        for (int k = 0; k < VW; ++k) {
            const uint64_t xb = (uint64_t)__double_as_longlong(x[k]);
            p[k] = WINDOW ? mul_rn_quick(ca, xb, far) : mul_rn_range(ca, xb, far);
        }
        if (WINDOW ? (int32_t)far < 0 : far >= ca.span) {
            const uint64_t ab = (uint64_t)__double_as_longlong(alpha);
#pragma unroll
            for (int k = 0; k < VW; k += 2) {  // out of line
                const ulonglong2 r = mul2_rn_hw_bits(ab, (uint64_t)__double_as_longlong(x[k]),
                                                     (uint64_t)__double_as_longlong(x[k + 1]));
                p[k] = r.x;
                p[k + 1] = r.y;
            }
        }
#pragma unroll
        for (int k = 0; k < VW; ++k) w[k] = __dadd_rn(__longlong_as_double((long long)p[k]), y[k]);
    } else {
        wxpy_vec_emu<VW, EMU>(alpha, x, y, w, base);
    }
}

#endif  // __CUDACC__

}  // namespace wx

#undef WX_EMU_FN
