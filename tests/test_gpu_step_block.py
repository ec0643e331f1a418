"""The block-per-instance step kernel at the edges of its tiles: 128-position groups of the queue, 32
horizon offsets and 32 workers per lane set, the lanes' lists of four largest keys, thread counts.
Whole numbers against the checker: the tolerance is equality."""
import numpy as np
import pytest

from paper_2605_06113_b200 import workload as wlm
from helpers import EMPTY, run_parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,B,W,H,kw", [
    (32, 8, 124, 15, dict()), (33, 8, 128, 31, dict()), (32, 16, 132, 32, dict(R_max=5)), (64, 8, 512, 63, dict()),
    (1, 8, 4, 80, dict()), (5, 72, 516, 3, dict(R_max=5)), (64, 64, 260, 8, dict(R_max=1)), (2, 256, 1024, 5, dict()),
    (33, 8, 640, 0, dict(R_max=5)), (1, 8, 132, 0, dict(threads=64)),
])
def test_tile_edges(G, B, W, H, kw):
    kw = dict(kw)
    threads = kw.pop("threads", 0)
    for term_mode, pred_mode, gate in ((1, 0, 0.5), (2, 0, 0.1), (3, 1, 0.5)):
        if H == 0 and term_mode != 1:
            continue
        cfg = wlm.get_config("c2", G=G, B=B, W=W, H=H, init_active=B - B // 8, init_queue=W - 1, hazard=0.05,
                             term_mode=term_mode, pred_mode=pred_mode, gate=gate, out_mu=2.0, score_mode=-1,
                             S_greedy=-1, delta_T=-1, arrival=("const", 6.0), **kw)
        run_parity(cfg, 2, 12, threads=threads, launch_steps=3, check_every=1)


@pytest.mark.parametrize("threads", [32, 96, 256])
@pytest.mark.parametrize("H,R_max", [(0, 5), (4, 5), (40, 4)])
@pytest.mark.parametrize("positions", [
    [5 + 32 * i for i in range(10)],                      # one router lane's (it reads every 32nd): its list of four runs dry
                                                          # while the window of five is built
    [37, 69, 101, 133] + [65 + 6 * i for i in range(6)],  # its list is used up by the window and runs dry after an admission
])
def test_one_lane_holds_the_whole_window(H, R_max, threads, positions, monkeypatch):
    make = wlm.make_workload

    def patched(*args, **kwargs):
        wl = make(*args, **kwargs)
        q = wl.state["wq_s"]
        for i, pos in enumerate(positions):
            q[:, pos] = 90000 - 7 * i
        return wl

    monkeypatch.setattr(wlm, "make_workload", patched)
    for S_greedy in (0, 1 << 20):
        cfg = wlm.get_config("c2", G=33, B=16, W=384, H=H, R_max=R_max, init_active=15, init_queue=380, hazard=0.05,
                             term_mode=1, S_greedy=S_greedy, score_mode=-1, delta_T=-1)
        run_parity(cfg, 2, 8, threads=threads, check_every=1)


@pytest.mark.parametrize("H", [0, 8, 40])
@pytest.mark.parametrize("W,n", [(128, 128), (256, 256), (260, 256), (128, 127)])
def test_every_request_beyond_the_peak(H, W, n, monkeypatch):
    # the queue fills whole groups of 128 positions, so no empty one ends the search for the largest request at or
    # below the peak of the score, and every request is above it (equal margins: the first admission's peak is zero)
    make = wlm.make_workload

    def patched(*args, **kwargs):
        wl = make(*args, **kwargs)
        st = wl.state
        run = st["act_base"] != EMPTY
        st["act_base"][...] = np.where(run, 500, EMPTY)
        st["load"][...] = 500 * run.sum(-1)
        st["wq_s"][:, :n] = 3000 + (np.arange(n) * 37) % 500
        return wl

    monkeypatch.setattr(wlm, "make_workload", patched)
    for S_greedy in (0, 1 << 20):
        cfg = wlm.get_config("c2", G=9, B=16, W=W, H=H, R_max=4, init_active=14, init_queue=n, hazard=0.05, term_mode=1,
                             S_greedy=S_greedy, score_mode=-1, delta_T=-1, arrival=("const", 0.0))
        for threads in (32, 128):
            run_parity(cfg, 2, 5, threads=threads, check_every=1)


@pytest.mark.parametrize("H", [0, 2])
def test_admissions_at_the_largest_positions_workers_and_counts(H):
    # the entry of an admission packs the queue position (4,096), the worker (64) and its free slots (256)
    cfg = wlm.get_config("c2", G=64, B=256, W=4096, H=H, R_max=5, init_active=230, init_queue=4096, hazard=0.02, term_mode=1,
                         score_mode=-1, S_greedy=600, delta_T=-1, arrival=("const", 30.0))
    run_parity(cfg, 1, 4, check_every=1)
    cfg = wlm.get_config("c2", G=64, B=256, W=4096, H=H, R_max=5, init_active=0, init_queue=4096, hazard=0.02, term_mode=1,
                         score_mode=-1, S_greedy=10, delta_T=-1, arrival=("const", 30.0))
    run_parity(cfg, 1, 2, check_every=1)


@pytest.mark.parametrize("hazard", [0.0, 0.01, 0.4, 1.0])
@pytest.mark.parametrize("G,B,W,H", [(33, 24, 128, 0), (5, 200, 64, 0), (16, 64, 128, 4), (64, 8, 64, 18), (3, 256, 64, 9), (40, 16, 64, 40)])
def test_single_warp_settles_endings_ahead_of_the_router(G, B, W, H, hazard):
    # none, one and several requests of a worker end at a step, in every word of its occupancy, admitted ones among them
    cfg = wlm.get_config("c2", G=G, B=B, W=W, H=H, init_active=B - B // 8, init_queue=W - 1, hazard=hazard, term_mode=1,
                         score_mode=-1, S_greedy=-1, delta_T=-1, arrival=("const", 9.0))
    run_parity(cfg, 2, 8, threads=32, launch_steps=2, check_every=1)


@pytest.mark.parametrize("G,H", [(5, 0), (33, 0), (33, 3), (16, 8), (40, 11), (7, 12), (33, 19), (3, 20), (34, 33)])
def test_score_matrix_of_every_horizon_group(G, H):
    # every number of offset groups and both numbers of workers per lane; the scores are compared for equality
    cfg = wlm.get_config("c2", G=G, B=16, W=132, H=H, init_active=14, init_queue=120, hazard=0.05, term_mode=1, score_mode=-1,
                         S_greedy=-1, delta_T=-1, arrival=("const", 4.0))
    run_parity(cfg, 2, 4, check_every=1, fscore=True)
