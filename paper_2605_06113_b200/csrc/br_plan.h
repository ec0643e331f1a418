// Decisions of the host side that need no CUDA: plain C++, so that they can be tested without a device.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace br {

constexpr int kMaxShared = 227 * 1024;     // dynamic shared memory of a thread block, at most
constexpr int kSharedPerSM = 227 * 1024;   // ... of the blocks of an SM together, with 1 KB more for each

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

// ---- launch shape of br_step_kernel ----------------------------------------------------------------

// Groups of four horizon offsets (h = 0 .. H) that a kernel unrolls: 2, 3 or 5, so that the loops over h
// of the admission loop are straight code; 0: a longer horizon, three offsets per lane, plain loops.
constexpr int step_groups(int H) { return H < 8 ? 2 : (H < 12 ? 3 : (H < 20 ? 5 : 0)); }

// Registers a thread of an instantiation may use, by Eq. 1 or 2 (fp) and step_groups(H).  The lean ones make the
// router's chain 5 to 15 % longer and let more instances be resident; horizons below 12 have none (at 80 registers
// 40 % more instances, each slower by as much: 2,072 of G = 16, H = 8, eight steps: 382 us, 396).  H = 12 to 19 at 96
// registers keeps values of the admission loop in memory: 1,184 of G = 8, H = 16, look-ahead, three steps 51.4 us, 46.9 at
// 112; of G = 48, B = 24, H = 12, classifier, 100.6, 80.9.  An SM holds 16 such warps, 20 of the lean ones: 2,960 of G = 8, H = 12
// 39.3 us, 29.6.
constexpr int step_register_cap(bool fp, int groups, bool lean)
{
    return !fp ? (lean ? 72 : 96) : groups == 5 ? (lean ? 96 : 112) : groups ? 96 : (lean ? 96 : 128);
}
// ... and the registers that it is compiled to, in the multiples of eight that an SM gives out (br_debug_step_registers
// compares them with the kernels).  Eq. 1: 75 and 79 for one worker per router lane, 80 for two, 87 where a single warp
// settles endings early; long horizons 111 and 114.
constexpr int step_registers(bool fp, int workers_per_lane, int groups, bool lean, bool early = false)
{
    return !fp ? (lean ? 72 : (workers_per_lane == 2 && early ? 88 : 80)) : groups == 5 ? (lean ? 96 : 112) : groups ? 96 : (lean ? 96 : (workers_per_lane == 1 ? 112 : 120));
}
constexpr bool step_has_lean(bool fp, int groups) { return !fp || !groups || groups == 5; }

// Warps of a kernel that an SM's registers hold: four partitions of 16,384, and 32 threads of a multiple of eight
// registers per warp (96 registers: 20 warps, not 21).
constexpr int step_warps_per_sm(int registers) { return 4 * (16384 / (32 * ((registers + 7) / 8 * 8))); }

struct StepShape {
    bool fp;               // Eq. 2
    int G, H, B, W;
    int term_mode, pred_mode;
    int shared;            // bytes of shared memory of an instance
};
struct StepLaunch { int warps; bool lean, early; };

// Whether a single warp settles the requests that end ahead of the router (constant hazard): with many instances
// resident it saves two trips to memory of each, which the router's chain would wait for: us per call of one step,
// 3,040 instances: G = 40, H = 0, W = 256: 26.9 -> 22.3, G = 64, W = 512: 45.6 -> 29.8, G = 48, H = 4: 165 -> 157.
// Instances of few slots and long horizons gain nothing.
inline bool step_early(const StepShape &s)
{
    return s.term_mode == 1 && (!s.fp || (step_groups(s.H) && s.G * s.B >= 512));
}

// ceil(2^32 / (B / 4)): the worker of slot quad q < 2^14 is the upper half of q times this (B / 4 <= 64, so the error
// stays below q * 64 < 2^32)
inline uint32_t quad_magic(int B) { return (uint32_t)(((1ull << 32) + B / 4 - 1) / (B / 4)); }

// log2 of the lanes per worker that turn its prediction buckets into L_g(k+h), of `threads`
inline int step_seg_log2(int G, int H, int threads)
{
    int q = 0;
    while (q < 5 && (G << (q + 1)) <= threads && (2 << q) <= H + 1) ++q;
    return q;
}

// Warps per instance, and which instantiation, for n_instances instances on `sms` SMs.
//
// More warps shorten an instance's parallel phases and leave fewer instances resident, so a batch of a few instances
// per SM takes as many warps as there is work for, a large one those that need the least time for all its
// waves.  With r resident instances of w warps a step takes, in units of the router's chain,
//     t(w, r) = 1 + 0.05 u(w) + p (c + e r) / w,
// u (H >= 20 alone; below, the router sums in registers) the offsets that a lane sums one after the other for L_g(k+h),
// each of which raises one word with the other workers (41 workers and 60 offsets: 60 each with two warps, 30 with three;
// 2,051 instances, H = 59, three steps: 162 and 131 us), p the thousands of slots that the projection streams (look-ahead,
// which reads no rows, half of it; more the longer the classifier's rows, above all where terminations read every
// row, two fifths more under the constant hazard where they are not whole vectors; Eq. 1 has draws and queue alone) and e what another
// resident instance costs.  The last, incomplete wave starts while instances of the one before still run and counts in part.
// The constants of Eq. 2 are a fit to 37,000 measured times (3,364 batches of 226 shapes, 20 to 4,500 instances, one to eight
// warps, both instantiations; full fleets, and fleets after some hundred steps), by terminations.  The choice is on average
// within 1.2 % of the fastest with look-ahead (at worst 13), 2.7 % under the constant hazard (5 in 100 more than 11), 3.3 %
// where terminations read every row (5 in 100 more than 20).  Neighbouring counts differ by up to a factor of two where rows
// fall out of the cache, which the estimate does not know: 1,455 of G = 29, B = 128, H = 34, three steps: 534 us at two warps, 348 at three.
// us per call at 1, 2, 3, 4, 5 warps: 1,036 of G = 64, W = 1,024, H = 8: 62 / 63 / 65 / 56 / 57; 1,332: 104 / 88 / 71 / 64 / 76;
// 2,960 of G = 15, W = 40, H = 19: 49 (41 lean) / 61 / 70 / 77 / 91; 1,036 of G = 24, B = 40, H = 12, terminations from rows: 79 /
// 55 / 67 / 67 / 84.  Four warps at least for instances that stream 4,096 slots with rows of 8 to 19, or half as many when
// terminations read every row: more of them resident take each other's cache lines (2,960 of G = 32, H = 11, terminations
// from rows: 428 / 255 / 203 / 193).
// Eq. 1 keeps its own older constants: within 2 % of the fastest on average over its usual shapes, 6 % over 364 batches of
// large fleets and queues, where routers of two- and four-warp blocks meet on the same partitions (1,006 of G = 54, B = 96,
// W = 888, four steps, 78 / 90 / 66 / 88 us at 1, 2, 3, 4 warps).
inline StepLaunch step_launch(const StepShape &s, int n_instances, int sms)
{
    const int groups = step_groups(s.H), A = s.G * s.B, n = (n_instances + sms - 1) / sms;
    const bool classifier = s.H > 0 && s.pred_mode == 0;
    int most = s.H > 0 ? A / 16 : 64;                      // threads with something to do: 16 slots, 4 positions, 8 offsets
    if (s.W / 4 > most) most = s.W / 4;
    if (s.G * (s.H + 1) / 8 > most) most = s.G * (s.H + 1) / 8;
    most = (most + 31) / 32;
    most = most < 4 ? 4 : (most > 8 ? 8 : most);
    const bool every_row = classifier && s.term_mode == 2, ragged = (s.H & 3) && s.H > 2;
    const bool long_rows = classifier && s.H >= 8 && groups && A * (every_row ? 2 : 1) >= 4096;
    const int least = long_rows ? 4 : 1;
    double p = 1e-3 * A;
    if (!s.H) p = 0.035 + 0.006 * s.G + 7e-5 * s.W;
    else if (every_row) p = p * (1.0 + 0.054 * s.H) + 7e-5 * s.W;
    else if (classifier) p = p * (1.0 + 0.025 * s.H) * (ragged ? 1.4 : 1.0) + 7e-5 * s.W;
    else p = 0.5 * p + 2e-4 * s.W;
    struct Fit { double c, e, last, last_full; };
    const Fit k = !s.H ? Fit{0.65, 0.03, 0.3, 0.4} : every_row ? Fit{0.34, 0.09, 0.47, 0.71}
                              : classifier ? Fit{0.65, 0.04, 0.45, 0.65} : Fit{0.39, 0.002, 0.27, 0.8};
    StepLaunch best = {1, false, false};
    double cost = 1e300;
    for (int w = least; w <= most; ++w) {
        double base = 1.0;
        if (s.H > 0 && !groups) {
            const int q = step_seg_log2(s.G, s.H, 32 * w);
            const int u = (((s.G << q) + 32 * w - 1) / (32 * w)) * ((s.H + (1 << q)) >> q);
            base += 0.05 * u * (s.G < 32 ? s.G : 32) / 32.0;
        }
        for (int lean = 0; lean < 2; ++lean) {
            // (the lean instantiation of H >= 20 spills in the classifier's loop, which a single warp cannot hide)
            if (lean && (!step_has_lean(s.fp, groups) || (classifier && !groups && w < 2))) continue;
            int r = step_warps_per_sm(step_registers(s.fp, s.G <= 32 ? 1 : 2, groups, lean != 0, w == 1 && step_early(s))) / w;
            const int fit = kSharedPerSM / (s.shared + 1024);
            if (r > fit) r = fit;
            if (r > 32) r = 32;
            if (r < 1) r = 1;
            const int full = n / r, part = n % r;
            double t = full * (base + p * (k.c + k.e * r) / w);
            if (part) t += (full ? k.last + k.last_full * part / r : 1.0) * (base + p * (k.c + k.e * part) / w);
            if (lean) t *= s.H ? 1.16 : 1.1;
            if (t <= cost) { cost = t; best.warps = w; best.lean = lean != 0; }
        }
    }
    best.early = best.warps == 1 && step_early(s);
    return best;
}

}  // namespace br
