"""Snapshots whose running counts say more free slots than the occupancy words have: flagged, no slot given twice, and
the envelope is that of the recorded loads."""
import numpy as np
import pytest
import torch

from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router, ST_BAD_STATE, state_to_numpy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,threads", [("c3", 32), ("c3", 64), ("c3", 128), ("c2", 32), ("c2", 128)])
@pytest.mark.parametrize("missing", [1, 5])
def test_occupied_slots_are_not_given_out(name, threads, missing):
    cfg = wlm.get_config(name, init_active=64, init_queue=200, hazard=0.0, term_mode=1, arrival=("const", 1.0))
    assert cfg.B == 64
    wl = wlm.make_workload(cfg, n_instances=3)
    r = Router(wl, device="cuda:0", threads=threads)
    st = r.device_state()
    st["nact"][:2] -= missing                     # two instances claim free slots that are all taken
    st["nact"][2, 1:] -= missing                  # the third also has a worker that is really full
    before = state_to_numpy(st)
    st["wq_s"][:] = 50000                         # one request turned away would lift the envelope
    out = r.outputs(3)
    probs = torch.zeros((1, 3, cfg.G, cfg.B, cfg.H), device="cuda:0") if cfg.H else None
    r.step(st, out, probs)
    a = out["assign"][0].cpu().numpy()
    load, trace, status = (out[k][0].cpu().numpy() for k in ("load", "trace", "status"))
    for i in range(3):
        assert status[i] & ST_BAD_STATE
        assert np.array_equal(trace[i], [load[i].max(), load[i].min(), load[i].sum()])
        assert (a[i] == -1).all()                 # every slot was taken
    after = state_to_numpy(st)
    assert np.array_equal(after["occ"], before["occ"]) and np.array_equal(after["act_base"], before["act_base"])
    r.close()
