"""The registers that a launch shape is chosen by are those of the kernels: 65,536 of an SM are given out to warps in units of
eight a thread, and a batch that is planned as one wave runs as two where the kernel needs more."""
import ctypes as C

import pytest

from paper_2605_06113_b200 import binding

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("early", [0, 1])
@pytest.mark.parametrize("lean", [0, 1])
@pytest.mark.parametrize("score_mode,H", [(0, 0), (1, 0), (1, 7), (1, 8), (1, 11), (1, 12), (1, 19), (1, 20), (1, 80)])
@pytest.mark.parametrize("G", [1, 32, 33, 64])
def test_planned_registers_are_the_kernels(score_mode, G, H, lean, early):
    planned = C.c_int32()
    used = binding.lib().br_debug_step_registers(score_mode, G, H, lean, early, C.byref(planned))
    assert used > 0 and (used + 7) // 8 * 8 == planned.value
