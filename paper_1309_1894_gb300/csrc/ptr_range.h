// ptr_range.h -- whether a kernel may read a caller's range of memory.
//
// A copy call looks up its source and refuses one that is not allocated or is
// shorter than the copy; a kernel that reads the same range faults, and the
// process loses its context.  So a range is handed to a kernel only if it lies
// inside one allocation of the kernel's device, and to the copy call otherwise.
// Plain host C++: the lookup is passed in.
#pragma once

#include <cstdint>

namespace wx {

// What is known of an address: the allocation it lies in.
struct AddressInfo {
    bool plain_device;  // device memory (not managed, not host memory), mapped
    int device;
    uint64_t start, size;  // of the allocation
};

// query(address, &info) is false where nothing is known.  The last byte is asked
// for too: an address range may be reserved beyond what is mapped of it.
template <class Query>
bool range_on_device(uint64_t p, uint64_t bytes, int device, Query query) {
    AddressInfo a{}, z{};
    if (bytes == 0 || p + (bytes - 1) < p) return false;
    if (!query(p, &a) || !query(p + (bytes - 1), &z)) return false;
    return a.plain_device && z.plain_device && a.device == device && z.device == device &&
           a.start == z.start && a.start <= p && p - a.start <= a.size &&
           bytes <= a.size - (p - a.start);
}

}  // namespace wx
