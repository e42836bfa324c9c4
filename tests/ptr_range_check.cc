// ptr_range_check.cc -- range_on_device (ptr_range.h) over a made-up address
// space, for the tests: allocations given as rows {first address mapped, bytes
// mapped, start reported, size reported, plain device memory, device}.
#include <cstdint>

#include "../paper_1309_1894_gb300/csrc/ptr_range.h"

extern "C" int range_check(const uint64_t (*rows)[6], int count, uint64_t p, uint64_t bytes,
                           int device) {
    return wx::range_on_device(p, bytes, device, [&](uint64_t a, wx::AddressInfo *info) {
        for (int i = 0; i < count; ++i) {
            const uint64_t *r = rows[i];
            if (a - r[0] >= r[1]) continue;
            *info = wx::AddressInfo{r[4] != 0, (int)r[5], r[2], r[3]};
            return true;
        }
        return false;
    });
}
