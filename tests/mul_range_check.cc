// mul_range_check.cc -- the integer-pipeline product over its whole range of
// operands (fp64_mul.cuh: mul_rn_range) against the host's own IEEE
// multiplication, for the tests.
#include <cstdint>
#include <cstring>

#include "../paper_1309_1894_gb300/csrc/fp64_mul.cuh"

static uint64_t bits(double v) {
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return u;
}

extern "C" {

// For i < n: away[i] is set when the pair left the fast path; returns the
// number of pairs on it whose bits differ from the host's product.
int64_t mul_range_check(int64_t n, double a, const double *b, uint8_t *away) {
    const wx::MulCoef c = wx::mul_coef_of(bits(a));
    int64_t bad = 0;
    for (int64_t i = 0; i < n; ++i) {
        uint32_t far = 0;
        const uint64_t r = wx::mul_rn_range(c, bits(b[i]), far);
        away[i] = far >= c.span;
        if (!away[i]) bad += r != bits(a * b[i]);
    }
    return bad;
}

// Whether a vector of products leaves the fast path.
int mul_range_any(int64_t n, double a, const double *b) {
    const wx::MulCoef c = wx::mul_coef_of(bits(a));
    uint32_t far = 0;
    for (int64_t i = 0; i < n; ++i) wx::mul_rn_range(c, bits(b[i]), far);
    return far >= c.span;
}

}  // extern "C"
