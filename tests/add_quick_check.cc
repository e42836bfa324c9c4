// add_quick_check.cc -- the windowed integer-pipeline sum (fp64_emu.cuh:
// add_rn_quick) against the host's own IEEE addition, for the tests.
#include <cstdint>
#include <cstring>

#include "../paper_1309_1894_gb300/csrc/fp64_emu.cuh"

static uint64_t bits(double v) {
    uint64_t u;
    std::memcpy(&u, &v, 8);
    return u;
}

// For i < n: away[i] is set when the pair left the fast path; returns the number
// of pairs on it whose bits differ from the host's sum.
extern "C" int64_t add_quick_check(int64_t n, const double *a, const double *b, uint8_t *away) {
    int64_t bad = 0;
    for (int64_t i = 0; i < n; ++i) {
        uint32_t w = 0;
        const uint64_t r = wx::add_rn_quick(bits(a[i]), bits(b[i]), w);
        away[i] = (uint8_t)(w >> 31);
        if (!away[i]) bad += r != bits(a[i] + b[i]);
    }
    return bad;
}
