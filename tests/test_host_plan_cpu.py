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
