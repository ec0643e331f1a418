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

// How a step uses an array of the snapshot or of its results: every row once, only the slots that change, or (the
// optional score matrix) every element by itself.
enum HostUse { kHostRows, kHostSparse, kHostScores };

// Whether a host-buffer step uses a page-locked array in place.  BR-0 reads and writes every row once, at the rate
// of the copy engines (50 GB/s measured either way), and of the sparse arrays only the slots that change (3 ns each
// against 150 ns for the 8 KB of an instance).  4,096 instances of G = 32, W = 256: 2.4 ms with every array copied
// both ways, 0.84 with only the sparse ones in place, 0.48 with all.  BR-H in large batches reads its snapshot
// and its classifier rows in smaller pieces than the bus likes and copies them; small batches save the
// copies' call time (16 instances: 147 us -> 47).  Terminations drawn from the classifier's output read every row in
// pieces, which costs more than those calls beyond about 100,000 slots (G = 64, H = 8, B = 64, us in place / copied:
// 224 / 276 at 16 instances, 456 / 380 at 40, 656 / 487 at 63; H = 16, B = 256: 294 / 382 at 4, 750 / 632 at 16).
// Scores go out eight bytes at a time: 1,024 instances of G = 32, W = 256: 19.4 ms in place, 2.0 copied.
inline bool host_in_place(HostUse use, int H, int term_mode, long long n_instances, long long slots_per_instance)
{
    if (use == kHostScores) return false;
    if (use == kHostSparse || (H == 0 && term_mode <= 1)) return true;
    return n_instances < 64 && (term_mode != 2 || n_instances * slots_per_instance <= 100000);
}

}  // namespace br
