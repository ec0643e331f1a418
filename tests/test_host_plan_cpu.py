"""Host-side decisions of the library (csrc/br_plan.h), compiled alone with the host compiler: no CUDA, no device."""
import ctypes as C
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_06113_b200", "csrc")

SHIM = r"""
#include "br_plan.h"
// page-locked ranges [start, start + size); the device sees host address x as x + shift
extern "C" uintptr_t alias(uintptr_t host, size_t bytes, int n, const uintptr_t *start, const size_t *size, const uintptr_t *shift)
{
    return br::device_alias(host, bytes, [&](uintptr_t at, br::LockedRange *r) {
        for (int i = 0; i < n; ++i)
            if (at >= start[i] && at - start[i] < size[i]) {
                r->dev = at + shift[i]; r->start = start[i] + shift[i]; r->size = size[i];
                return true;
            }
        return false;
    });
}
extern "C" int launch(int fp, int G, int H, int B, int W, int term_mode, int pred_mode, int shared, int n, int *resident)
{
    const br::StepShape s = {fp != 0, G, H, B, W, term_mode, pred_mode, shared};
    const br::StepLaunch l = br::step_launch(s, n, 148);
    *resident = br::step_warps_per_sm(br::step_registers(s.fp, G <= 32 ? 1 : 2, br::step_groups(H), l.lean)) / l.warps;
    return l.lean ? -l.warps : l.warps;
}
extern "C" uint32_t magic(int B) { return br::quad_magic(B); }
extern "C" int in_place(int use, int H, int term_mode, long long n, long long slots)
{
    return br::host_in_place((br::HostUse)use, H, term_mode, n, slots);
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "libplan.so")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC, "-o", so, str(d / "shim.cpp")])
    return C.CDLL(so)


def _alias(plan, host, nbytes, ranges):
    n = len(ranges)
    arrays = [(t * n)(*(r[i] for r in ranges)) for i, t in enumerate((C.c_size_t, C.c_size_t, C.c_size_t))]
    plan.alias.restype = C.c_size_t
    return plan.alias(C.c_size_t(host), C.c_size_t(nbytes), n, *arrays)


def test_arrays_are_used_in_place_only_where_every_byte_is_page_locked(plan):
    P = 4096
    base = 1 << 40
    one = [(base, 8 * P, 0)]
    assert _alias(plan, base, 8 * P, one) == base
    assert _alias(plan, base + 16, 8 * P - 16, one) == base + 16
    assert _alias(plan, base + 8, 16, one) == 0                                   # not aligned
    assert _alias(plan, base, 0, one) == 0
    assert _alias(plan, base, 8 * P + 1, one) == 0                                # runs over the end
    assert _alias(plan, base - 16, 32, one) == 0                                  # starts before it
    # both ends page-locked, pages in between not
    assert _alias(plan, base, 8 * P, [(base, 2 * P, 0), (base + 6 * P, 2 * P, 0)]) == 0
    assert _alias(plan, base + P, 6 * P, [(base, 2 * P, 0), (base + 6 * P, 2 * P, 0)]) == 0
    # one array over adjacent registrations, contiguous on the device or not
    assert _alias(plan, base + P, 6 * P, [(base, 2 * P, 64), (base + 2 * P, 6 * P, 64)]) == base + P + 64
    assert _alias(plan, base + P, 6 * P, [(base, 2 * P, 0), (base + 2 * P, 6 * P, P)]) == 0
    assert _alias(plan, base, 16, [(base, P, 8)]) == 0                            # the device address is not aligned


def test_which_page_locked_arrays_are_used_in_place(plan):
    rows, sparse, scores = 0, 1, 2

    def in_place(use, H, term, n, slots):
        return bool(plan.in_place(use, H, term, C.c_longlong(n), C.c_longlong(slots)))

    for H, term, n, slots in ((0, 1, 1, 2048), (0, 0, 4096, 2048), (8, 2, 40, 4096), (80, 3, 4096, 512)):
        assert not in_place(scores, H, term, n, slots)          # an element at a time over the bus
        assert in_place(sparse, H, term, n, slots)
    assert in_place(rows, 0, 1, 4096, 4096) and in_place(rows, 8, 1, 63, 16384) and in_place(rows, 80, 3, 63, 16384)
    assert not in_place(rows, 8, 1, 64, 64) and not in_place(rows, 0, 3, 64, 64)
    # terminations drawn from every classifier row
    assert in_place(rows, 8, 2, 24, 4096) and not in_place(rows, 8, 2, 25, 4096) and not in_place(rows, 16, 2, 63, 16384)


def _launch(plan, G, H, n, B=64, W=256, term=1, pred=0, shared=8000):
    res = C.c_int()
    w = plan.launch(int(H > 0), G, H, B, W, term, pred, shared, n, C.byref(res))
    return abs(w), w < 0, min(res.value, 232448 // (shared + 1024))


def test_registers_hold_whole_partitions_of_warps(plan):
    # 96 registers: five warps on each of four partitions
    assert _launch(plan, 32, 8, 148 * 10)[2] == 10 and _launch(plan, 32, 8, 148 * 7)[2] >= 7


def test_a_batch_is_not_split_into_waves_that_fewer_warps_would_save(plan):
    # one wave of two warps, not two of three or more (7 and 10 instances an SM), nor two of two where one warp each
    # makes one (14)
    for G, H, B in ((32, 1, 64), (16, 4, 64), (16, 8, 64), (4, 2, 24)):
        for n in (7, 10):
            w, _, res = _launch(plan, G, H, 148 * n, B=B)
            assert w == 2 and res >= n, (G, H, n)
    assert _launch(plan, 4, 2, 148 * 14, B=24, W=32)[0] == 1
    assert _launch(plan, 32, 1, 148 * 5)[0] == 4 and _launch(plan, 32, 1, 148 * 4)[0] >= 4
    # two full waves of two warps, not a full and a nearly empty one of a single warp
    assert _launch(plan, 20, 12, 3000, B=96, shared=12000)[0] == 2
    # batches that just miss a wave take the lean instantiation where there is one
    assert _launch(plan, 40, 0, 148 * 28, shared=6000) == (1, True, 28)
    assert _launch(plan, 7, 60, 148 * 19, W=32, term=3, pred=1, shared=8000)[:2] == (1, True)
    # three warps split the offsets of 41 workers, two do not
    assert _launch(plan, 41, 59, 1738, B=24, W=84, term=3, pred=1, shared=27000)[:2] == (3, True)
    # long classifier rows: four or five warps whatever the batch
    for n in (4, 7, 10, 14, 20, 28):
        assert _launch(plan, 64, 8, 148 * n, shared=20000)[0] in (4, 5)


def test_every_shape_gets_a_launch(plan):
    for G in (1, 2, 32, 33, 64):
        for H in (0, 1, 8, 19, 20, 80):
            for B, W in ((8, 4), (64, 1024), (256, 4096)):
                for term, pred in ((1, 0), (2, 0), (3, 0), (3, 1)):
                    if (term == 2 or pred) and H == 0:
                        continue
                    for n in (1, 148, 149, 4096, 1 << 20):
                        for shared in (4000, 60000, 232448):
                            w, _, res = _launch(plan, G, H, n, B, W, term, pred, shared)
                            assert 1 <= w <= 8


def test_the_worker_of_a_slot_quad(plan):
    plan.magic.restype = C.c_uint32
    for B in range(8, 257, 8):
        m = plan.magic(B)
        for q in range(64 * B // 4):                       # every quad of the largest fleet
            assert (q * m) >> 32 == q // (B // 4), (B, q)
