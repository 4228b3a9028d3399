// Whether a host array may be read in place by a kernel that nobody asked for
// (host code without CUDA, so that it can be tested anywhere).
#pragma once

#include <cstddef>
#include <cstdint>

namespace sr {

// What the driver says about one host address.
struct HostRange {
    bool page_locked = false;  // allocated or registered as page-locked, and mapped for the device
    uintptr_t start = 0;       // that one allocation or registration
    size_t size = 0;
    uintptr_t device = 0;      // the address's device address
};

// [x, x + bytes) (bytes > 0) lies in ONE page-locked allocation or registration that is
// mapped without a break.  The ends alone do not show it: between two registrations there
// may be ordinary memory, which a copy takes and a kernel may not read.
template <class Query> inline bool one_page_locked_range(uintptr_t x, size_t bytes, Query&& query) {
    const HostRange a = query(x);
    if (!a.page_locked || x < a.start || a.size < bytes || x - a.start > a.size - bytes) return false;
    const HostRange b = query(x + (bytes - 1));
    return b.page_locked && b.start == a.start && b.device - a.device == bytes - 1;
}

}  // namespace sr
