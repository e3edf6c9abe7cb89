// How far the memory behind a pointer is allocated, asked of the driver before
// a copy kernel writes there.  cudaMemcpyAsync refuses a range that runs past
// its allocation; a kernel would fault, so the copies that a kernel makes need
// the same refusal on the host.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace fasgd {

enum Reach {
    kReachUnknown = 0,    // the driver knows no allocation at p
    kReachOne = 1,        // one allocation holds [p, p + bytes)
    kReachSeveral = 2,    // neighbouring allocations or mappings do
    kReachShort = 3,      // memory ends before p + bytes
};

// find(p, &base, &size): the allocation that holds p; false if there is none.
template <class Find>
Reach reach(uintptr_t p, size_t bytes, Find find) {
    uintptr_t base = 0;
    size_t size = 0;
    if (!find(p, &base, &size) || p < base || p - base >= size) return kReachUnknown;
    if (size - (p - base) >= bytes) return kReachOne;
    size_t left = bytes - (size - (p - base));
    for (p = base + size; find(p, &base, &size) && base == p && size > 0; p += size) {
        if (size >= left) return kReachSeveral;
        left -= size;
    }
    return kReachShort;
}

}  // namespace fasgd
