"""Contexts used from different host threads at the same time, one context per thread: the launches of one must not
depend on those of another."""
import threading

import pytest
import torch

from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router

pytestmark = pytest.mark.gpu

STEPS = 10000         # a launch is refused in one of some hundred to a thousand where the limits race


def test_contexts_with_different_shared_memory_step_side_by_side():
    # one kernel (two workers a lane, long horizon), three amounts of shared memory beyond the default 48 KB
    routers = []
    for G, W in ((64, 4096), (56, 2048), (48, 2048)):
        cfg = wlm.get_config("h80", G=G, W=W, B=8, init_active=8, init_queue=8)
        wl = wlm.make_workload(cfg, n_instances=1)
        r = Router(wl, device="cuda:0")
        routers.append((r, r.device_state(), r.outputs(1), torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(len(routers))

    def work(r, st, out, stream):
        start.wait()
        try:
            call = r.prepare(st, out, stream=stream)
            for _ in range(STEPS):
                call()
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=x) for x in routers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for r, st, _, _ in routers:
        assert int(st["step"][0]) == STEPS
        r.close()
