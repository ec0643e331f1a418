"""Refreshes of c_hat from classifier rows of every width that is loaded as a whole (8, 4, 2 probabilities, or one by one) and
of every horizon group, with lists of due requests that fill their warp's part, run over a round of rows or
stay empty.  Whole numbers and fp32 c_hat against the checker: the tolerance is equality."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router
from helpers import run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [0, 32, 256])
@pytest.mark.parametrize("G,B,H,delta_T", [
    (3, 8, 1, 1), (5, 24, 2, 1), (21, 40, 6, 3), (7, 40, 7, 1), (9, 64, 4, 2), (16, 64, 8, 1), (40, 64, 8, 4), (11, 72, 9, 2),
    (6, 64, 11, 5), (6, 64, 12, 1), (5, 40, 16, 1), (40, 24, 18, 9), (3, 40, 20, 1), (2, 256, 27, 13),
])
def test_rows_of_every_width(G, B, H, delta_T, threads):
    for gate, active in ((0.02, B), (0.5, B - B // 4)):
        cfg = wlm.get_config("c2", G=G, B=B, W=64, H=H, init_active=active, init_queue=60, hazard=0.03, term_mode=1, gate=gate,
                             delta_T=delta_T, score_mode=-1, S_greedy=-1, arrival=("const", 3.0))
        run_parity(cfg, 3, 6, threads=threads, launch_steps=2, check_every=1)


@pytest.mark.parametrize("H", [2, 3, 8, 12, 27])
def test_rows_written_by_the_kernel_ahead(H):
    # rows that a kernel of the same stream writes directly before each step, different ones every time, nothing waiting for the
    # host in between
    cfg = wlm.get_config("c2", G=21, B=40, W=64, H=H, init_active=40, init_queue=60, hazard=0.0, term_mode=2, gate=0.1, delta_T=1,
                         score_mode=-1, S_greedy=-1, arrival=("const", 3.0))
    n, steps = 40, 12
    wl = wlm.make_workload(cfg, n_instances=n)
    r = Router(wl, device="cuda:0")
    st, out = r.device_state(), [r.outputs(n) for _ in range(steps)]
    rows = [wlm.term_probs_np(wl, k) for k in range(steps)]
    src = torch.from_numpy(np.stack(rows)).cuda()
    buf = torch.full(src.shape[1:], 0.9, device="cuda")
    torch.cuda.synchronize()
    for k in range(steps):
        torch.mul(src[k], 1.0, out=buf)
        r.step(st, out[k], buf)
    torch.cuda.synchronize()
    orcs = [oracle.instance_from_workload(wl, i) for i in range(n)]
    for k in range(steps):
        for i, o in enumerate(orcs):
            a, l, t, _ = o.step(rows[k][i])
            assert np.array_equal(out[k]["assign"][0, i].cpu().numpy(), a), (k, i)
            assert np.array_equal(out[k]["load"][0, i].cpu().numpy(), l) and np.array_equal(out[k]["trace"][0, i].cpu().numpy(), t), (k, i)
    r.close()
