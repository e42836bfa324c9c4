// fp64_mul.cuh -- IEEE 754 binary64 multiplication, round to nearest even,
// computed in the integer pipelines (the companion of fp64_emu.cuh's
// addition, for kernels with several products per element).
#pragma once

#include <cstdint>

// The cores (mul_coef_of, mul_rn_core, sqr_rn_core) also compile as plain
// host C++, so the host can check them against its own IEEE multiply.
#ifdef __CUDACC__
#define WX_MUL_FN __host__ __device__ __forceinline__
#else
#define WX_MUL_FN inline
#endif

namespace wx {

#ifdef __CUDACC__
static __device__ __noinline__ uint64_t mul_rn_hw_bits(uint64_t ua, uint64_t ub) {
    return (uint64_t)__double_as_longlong(
        __dmul_rn(__longlong_as_double((long long)ua), __longlong_as_double((long long)ub)));
}

// RN(a * b) and RN(a * c), one call for the two.
static __device__ __noinline__ ulonglong2 mul2_rn_hw_bits(uint64_t ua, uint64_t ub, uint64_t uc) {
    const double a = __longlong_as_double((long long)ua);
    return make_ulonglong2(
        (uint64_t)__double_as_longlong(__dmul_rn(a, __longlong_as_double((long long)ub))),
        (uint64_t)__double_as_longlong(__dmul_rn(a, __longlong_as_double((long long)uc))));
}
#endif

// Bits sh .. sh + 31 of the 64-bit word hi:lo, 0 <= sh < 32.
WX_MUL_FN uint32_t funnel_r(uint32_t lo, uint32_t hi, uint32_t sh) {
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, sh);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> sh);
#endif
}

// The same for any sh, with no bits left of the word at 32 and more.
WX_MUL_FN uint32_t funnel_rc(uint32_t lo, uint32_t hi, uint32_t sh) {
#ifdef __CUDA_ARCH__
    return __funnelshift_rc(lo, hi, sh);
#else
    return (uint32_t)((((uint64_t)hi << 32) | lo) >> (sh < 32u ? sh : 32u));
#endif
}

// RN(a * b) in the integer pipelines (multiply-adds on the FMA pipeline, the
// rest on the ALU).
//
// Method (the definition of a correctly rounded product).  For normal
// operands, split each 53-bit significand (hidden bit included) into a 21-bit
// high and a 32-bit low limb; four 32x32-bit products give the exact 106-bit
// product P = top 2^64 + w1 2^32 + w0, with P in [2^104, 2^106) and t = 1 when
// P >= 2^105.  The unrounded significand M is P >> (52 + t); g holds the 32
// bits of P below it.  Adding 2^31 to g carries into M exactly when the
// discarded part is at least one half, and g becomes 0 exactly when its own 32
// bits are one half: the discarded part is then one half if w0 is 0 as well
// (g reaches into w0, so the bits of w0 below g are zero exactly when w0 is),
// and that tie goes to even by clearing the lowest bit of the rounded-up M.
// The biased exponent is ea + eb - 1023 + t.  The result is assembled by
// adding M, hidden bit included, to sign | (exponent - 1) << 52, so a rounding
// carry to 2^53 lands in the exponent field by itself.

// One operand split once for many products (a coefficient: prepared on the
// host, read from the kernel's parameter space by every product).
struct MulCoef {
    uint32_t hi;   // high significand limb with the hidden bit (21 bits)
    uint32_t lo;   // low significand limb (32 bits)
    int32_t e;     // biased exponent - 1024; 2^20 when the operand is not normal
    uint32_t k;    // sign << 31 plus (biased exponent - 1024) << 20, modulo 2^32
    uint32_t win;  // mul_rn_quick: first exponent field of the other operand's window, << 21
    uint32_t from, span;  // mul_rn_range: first exponent field of the other operand's
                          // range, << 21, and the range's length, << 21 (0: none)
};

// The exponent window of mul_rn_quick: the 1024 exponent fields from first on,
// every one of which gives a product in the normal range whatever t and the
// rounding; 0 when the coefficient has no such window (it is not normal, or
// 2^1021 or more in magnitude).  The window starts as near to 512 (values from
// 2^-511) as the coefficient's exponent allows.
WX_MUL_FN int mul_window_first(uint64_t ua) {
    const int ea = (int)((ua >> 52) & 0x7FFu);
    if (ea == 0 || ea == 0x7FF) return 0;
    const int lo = 1024 - ea > 1 ? 1024 - ea : 1;               // result exponent field >= 1
    const int top = 0x7FB + 1024 - ea;                          // .. and <= 0x7FD with t = 1
    const int hi = (top < 0x7FE ? top : 0x7FE) - 1023;
    if (lo > hi) return 0;
    return lo > 512 ? lo : hi < 512 ? hi : 512;
}

WX_MUL_FN MulCoef mul_coef_of(uint64_t ua) {
    const uint32_t ah = (uint32_t)(ua >> 32);
    const uint32_t ea = (ah >> 20) & 0x7FFu;
    MulCoef c;
    c.hi = (ah & 0xFFFFFu) | 0x100000u;
    c.lo = (uint32_t)ua;
    c.e = ea - 1u >= 0x7FEu ? (1 << 20) : (int32_t)ea - 1024;
    c.k = (ah & 0x80000000u) + ((uint32_t)((int32_t)ea - 1024) << 20);
    c.win = (uint32_t)mul_window_first(ua) << 21;
    // result exponent fields 1 .. 0x7FD, t = 1 included, of normal operands
    const int32_t first = c.e < 0 ? -c.e : 1, last = c.e > -3 ? 0x7FB - c.e : 0x7FE;
    c.from = (uint32_t)first << 21;
    c.span = last >= first ? (uint32_t)(last + 1 - first) << 21 : 0u;
    return c;
}

// Rounds the 106-bit product top:w1:w0 and adds it to base (sign and exponent
// field - 1 - t); *t_out is t.
WX_MUL_FN uint64_t round_product(uint64_t top, uint32_t w1, uint32_t w0, uint32_t base,
                                 uint32_t *t_out) {
    const uint32_t tl = (uint32_t)top, th = (uint32_t)(top >> 32);
    const uint32_t sh = (th >> 9) + 20u;  // 20 + t: bit 105 of P is bit 9 of th
    const uint32_t ml = funnel_r(w1, tl, sh);
    const uint32_t mh = funnel_r(tl, th, sh);  // < 2^21, hidden bit at bit 20
    const uint32_t g = funnel_r(w0, w1, sh);
    const uint32_t hw = (base - (20u << 20)) + (sh << 20) + mh;
    uint32_t gs, lo, hi;
#ifdef __CUDA_ARCH__
    asm("add.cc.u32 %0, %3, 0x80000000;\n\t"
        "addc.cc.u32 %1, %4, 0;\n\t"
        "addc.u32 %2, %5, 0;"
        : "=r"(gs), "=r"(lo), "=r"(hi)
        : "r"(g), "r"(ml), "r"(hw));
#else
    gs = g + 0x80000000u;
    lo = ml + (g >> 31);
    hi = hw + (uint32_t)(lo < ml);
#endif
    lo = (gs | w0) == 0u ? lo & ~1u : lo;
    *t_out = sh - 20u;
    return ((uint64_t)hi << 32) | lo;
}

// The fast path of RN(c * b): the result's bits, and `slow` set when the
// operands or the result leave it (the bits are then meaningless): operands
// that are zero, subnormal, infinite or NaN, and products whose unrounded
// exponent field leaves [1, 0x7FD] (a subnormal, or a possible overflow).
WX_MUL_FN uint64_t mul_rn_core(const MulCoef &c, uint64_t ub, bool &slow) {
    const uint32_t bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
    const uint32_t eb = (bh >> 20) & 0x7FFu;
    const uint32_t b1 = (bh & 0xFFFFFu) | 0x100000u;
    const uint64_t p00 = (uint64_t)c.lo * bl;
    const uint64_t x = (uint64_t)c.hi * bl + (uint64_t)c.lo * b1 + (p00 >> 32);  // < 2^55
    const uint64_t top = (uint64_t)c.hi * b1 + (x >> 32);                        // < 2^42
    uint32_t t;
    // sign and exponent: the two signs add modulo 2 in bit 31
    const uint64_t bits =
        round_product(top, (uint32_t)x, (uint32_t)p00, c.k + (bh & 0xFFF00000u), &t);
    const int32_t ebase = c.e + (int32_t)(eb + t);  // result exponent - 1
    slow = slow || (eb - 1u >= 0x7FEu) || ((uint32_t)ebase >= 0x7FDu);
    return bits;
}

// The same product with the cheapest range check, for kernels whose products
// set the pace: ORs into `away` a word whose top bit is set when b's exponent
// field lies outside the coefficient's window (mul_window_first; zeros,
// subnormals, infinities and NaN always do, since a window lies in
// [1, 0x7FE]); the bits are then meaningless.  The coefficient must have a
// window.
WX_MUL_FN uint64_t mul_rn_quick(const MulCoef &c, uint64_t ub, uint32_t &away) {
    const uint32_t bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
    const uint32_t b1 = (bh & 0xFFFFFu) | 0x100000u;
    away |= (bh << 1) - c.win;
    const uint64_t p00 = (uint64_t)c.lo * bl;
    const uint64_t x = (uint64_t)c.hi * bl + (uint64_t)c.lo * b1 + (p00 >> 32);
    const uint64_t top = (uint64_t)c.hi * b1 + (x >> 32);
    uint32_t t;
    return round_product(top, (uint32_t)x, (uint32_t)p00, c.k + (bh & 0xFFF00000u), &t);
}

// How far b's exponent field lies above the first of the range of operands whose
// product with the coefficient is in the normal range whatever t and the rounding
// (modulo 2^32, so a field below it is far as well); c.span or more: outside.
WX_MUL_FN uint32_t mul_distance(const MulCoef &c, uint64_t ub) {
    return ((uint32_t)(ub >> 32) << 1) - c.from;
}

// The same product over that whole range: `far` becomes the largest distance so
// far, and the products made are meaningless once it is c.span or more.
WX_MUL_FN uint64_t mul_rn_range(const MulCoef &c, uint64_t ub, uint32_t &far) {
    const uint32_t bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
    const uint32_t b1 = (bh & 0xFFFFFu) | 0x100000u;
    // mul_distance(c, ub), from the word at hand: by way of ub the compiler orders the
    // wide maxpy groups another way, which is 2 % slower (GB300)
    const uint32_t d = (bh << 1) - c.from;
    far = d > far ? d : far;
    const uint64_t p00 = (uint64_t)c.lo * bl;
    const uint64_t x = (uint64_t)c.hi * bl + (uint64_t)c.lo * b1 + (p00 >> 32);
    const uint64_t top = (uint64_t)c.hi * b1 + (x >> 32);
    uint32_t t;
    return round_product(top, (uint32_t)x, (uint32_t)p00, c.k + (bh & 0xFFF00000u), &t);
}

// RN(a * b) of two data operands, with a cheap range check: `slow` is set when
// either exponent field is outside [512, 1534] (magnitudes 2^-511 up to 2^512),
// where every product is in the normal range.
WX_MUL_FN uint64_t mul_rn_quick2(uint64_t ua, uint64_t ub, bool &slow) {
    const uint32_t ah = (uint32_t)(ua >> 32), al = (uint32_t)ua;
    const uint32_t bh = (uint32_t)(ub >> 32), bl = (uint32_t)ub;
    const uint32_t a1 = (ah & 0xFFFFFu) | 0x100000u, b1 = (bh & 0xFFFFFu) | 0x100000u;
    slow |= ((ah << 1) - (512u << 21) >= (1023u << 21)) | ((bh << 1) - (512u << 21) >= (1023u << 21));
    const uint64_t p00 = (uint64_t)al * bl;
    const uint64_t x = (uint64_t)a1 * bl + (uint64_t)al * b1 + (p00 >> 32);
    const uint64_t top = (uint64_t)a1 * b1 + (x >> 32);
    uint32_t t;
    return round_product(top, (uint32_t)x, (uint32_t)p00,
                         (ah & 0xFFF00000u) + (bh & 0xFFF00000u) - (1024u << 20), &t);
}

// RN(a * a): both operands one value, so the split is taken once and the two
// cross products are one, doubled: P = A1^2 2^64 + 2 A1 A0 2^32 + A0^2 for the
// limbs A1 (21 bits, hidden bit included) and A0 (32 bits).  The sign is
// always clear, so the top word of the result tells by itself whether the
// exponent field left [1, 0x7FD]: 2 ea - 1024 + t runs from -1024 (zero,
// subnormal) to 3071 (infinity, NaN), which as a field of 12 bits names each
// value once, and the hidden bit adds one to it.  `slow` as in mul_rn_core.
WX_MUL_FN uint64_t sqr_rn_core(uint64_t ua, bool &slow) {
    const uint32_t ah = (uint32_t)(ua >> 32), a0 = (uint32_t)ua;
    const uint32_t a1 = (ah & 0xFFFFFu) | 0x100000u;
    const uint64_t p00 = (uint64_t)a0 * a0;
    const uint64_t x = (uint64_t)(a1 << 1) * a0 + (p00 >> 32);  // < 2^55
    const uint64_t top = (uint64_t)a1 * a1 + (x >> 32);           // P >> 64, < 2^42
    uint32_t t;
    const uint64_t bits = round_product(top, (uint32_t)x, (uint32_t)p00,
                                        ((ah << 1) & 0xFFE00000u) - (1024u << 20), &t);
    slow = slow || (uint32_t)(bits >> 32) - 0x100000u >= 0x7FD00000u;
    return bits;
}

#ifdef __CUDACC__
__device__ __forceinline__ uint64_t sqr_rn_bits(uint64_t ua) {
    bool slow = false;
    uint64_t bits = sqr_rn_core(ua, slow);
    if (slow) bits = mul_rn_hw_bits(ua, ua);
    return bits;
}

// RN(a * b) on two bit patterns, the hardware instruction out of line for the
// cases the fast path leaves out.
__device__ __forceinline__ uint64_t mul_rn_bits(uint64_t ua, uint64_t ub) {
    bool slow = false;
    uint64_t bits = mul_rn_core(mul_coef_of(ua), ub, slow);
    if (slow) bits = mul_rn_hw_bits(ua, ub);
    return bits;
}

#endif  // __CUDACC__

}  // namespace wx

#undef WX_MUL_FN
