// mul_quick_check.cc -- the windowed integer-pipeline products (fp64_mul.cuh:
// mul_rn_quick with a split coefficient, mul_rn_quick2 with two data operands)
// against the host's own IEEE multiplication, for the tests.
#include <cstdint>
#include <cstring>

#include "../paper_1309_1894_gb300/csrc/fp64_mul.cuh"

static uint64_t bits(double v) {
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return u;
}

extern "C" {

int mul_window(double a) { return wx::mul_window_first(bits(a)); }

// For i < n: away[i] is set when the pair left the fast path; returns the
// number of pairs on it whose bits differ from the host's product.
int64_t mul_quick_check(int64_t n, const double *a, const double *b, int two, uint8_t *away) {
    int64_t bad = 0;
    for (int64_t i = 0; i < n; ++i) {
        uint32_t w = 0;
        bool slow = false;
        const uint64_t r = two ? wx::mul_rn_quick2(bits(a[i]), bits(b[i]), slow)
                               : wx::mul_rn_quick(wx::mul_coef_of(bits(a[i])), bits(b[i]), w);
        away[i] = slow || (int32_t)w < 0;
        if (!away[i]) bad += r != bits(a[i] * b[i]);
    }
    return bad;
}

}  // extern "C"
