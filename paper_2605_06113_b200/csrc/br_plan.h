// Decisions of the host side that need no CUDA: plain C++, so that they can be tested without a device.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace br {

constexpr int kMaxShared = 227 * 1024;     // dynamic shared memory of a thread block, at most

// A page-locked allocation or registration around an address, in the device's address space.
struct LockedRange {
    uintptr_t dev;         // device address of the address asked for
    uintptr_t start;       // device address of the range
    size_t size;
};

// Device address of a host array that the kernels can use in place (every byte page-locked, contiguous on the
// device, 16-byte aligned), or 0.  lookup(address, range) says whether an address is page-locked.  Arrays are
// followed from range to range: two page-locked ends say nothing of the pages between them, and one
// array may be covered by several registrations.
template <typename Lookup>
inline uintptr_t device_alias(uintptr_t host, size_t bytes, Lookup lookup)
{
    if (!bytes || (host & 15)) return 0;
    uintptr_t dev = 0;
    for (size_t at = 0; at < bytes;) {
        LockedRange r;
        if (!lookup(host + at, &r) || r.dev < r.start || r.dev - r.start >= r.size) return 0;
        if (at == 0) dev = r.dev;
        else if (r.dev - dev != at) return 0;
        at += r.size - (r.dev - r.start);
    }
    return dev & 15 ? 0 : dev;
}

}  // namespace br
