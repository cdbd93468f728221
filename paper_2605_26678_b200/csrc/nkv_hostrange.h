// Which host memory the device may read where it lies.  Plain C++, so that the decision can be tested without a device.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace nkv {

// What the driver says about a host address: the device's address of it (null: none), and the allocation or registration
// that holds it, in the device's addresses.
struct HostRange {
    const unsigned char* device;
    uintptr_t start;
    size_t size;
};

// The device's address of [p, p + bytes), or null unless one allocation or registration holds all of it.  (With unified
// addressing the device's address of every pinned byte is its host address: two registrations that hold the first and the
// last byte say nothing about the pages in between.)  query(p, &range): false where the driver has no answer.
template <class Query>
const void* readable_in_place(const void* p, size_t bytes, Query&& query) {
    HostRange r = {nullptr, 0, 0};
    if (!p || bytes == 0 || !query(p, &r) || !r.device) return nullptr;
    const uintptr_t at = reinterpret_cast<uintptr_t>(r.device);
    if (at < r.start || at - r.start > r.size || bytes > r.size - (at - r.start)) return nullptr;
    return r.device;
}

}  // namespace nkv
