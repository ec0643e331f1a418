"""br_step_host on page-locked buffers, which the kernels use in place, on pageable ones, which are copied, and on a
mixture: state and outputs equal those of br_step on device buffers."""
import time

import numpy as np
import pytest
import torch

from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n_inst,kw", [("c3", 1, {}), ("c3", 63, {}), ("c3", 700, {}), ("c3", 540, dict(G=40, W=520)), ("c2", 3, {}),
                                            ("c2", 520, {}), ("c3", 70, dict(term_mode=3)), ("h80", 63, {}), ("h80", 64, {})])
@pytest.mark.parametrize("pinned", ["all", "some", "misaligned"])
def test_in_place_matches_device_step(name, n_inst, kw, pinned):
    cfg = wlm.get_config(name, **kw)
    wl = wlm.make_workload(cfg, n_instances=n_inst)
    r = Router(wl, device="cuda:0")

    def host(key, v):
        v = v.cpu()
        if pinned == "some" and key in ("wq_s", "trace", "act_base"):
            return v
        if pinned == "misaligned" and key in ("wq_id", "load", "act_id"):
            buf = torch.empty(v.numel() * v.element_size() + 8, dtype=torch.uint8).pin_memory()
            w = buf[8:].view(v.dtype).view(v.shape)
            w.copy_(v)
            return w
        return v.pin_memory()

    st_d, out_d = r.device_state(), r.outputs(n_inst)
    st_h = {k: host(k, v) for k, v in st_d.items()}
    out_h = {k: host(k, v) for k, v in out_d.items()}
    moved = []
    for k in range(3):
        probs = torch.from_numpy(np.ascontiguousarray(wlm.term_probs_np(wl, k))) if cfg.H > 0 and cfg.pred_mode == 0 else None
        moved.append(sum(r.step_host(st_h, out_h, None if probs is None else host("probs", probs))))
        r.step(st_d, out_d, None if probs is None else probs.cuda())
        torch.cuda.synchronize()
        for a, b in ((out_h, out_d), (st_h, st_d)):
            for key in a:
                if cfg.pred_mode == 1 and key in ("act_chat0", "act_kref"):
                    continue                      # not part of a snapshot with known lifetimes: the host step leaves them alone
                assert torch.equal(a[key], b[key].cpu()), (k, key)
    # act_id of page-locked snapshots stays where it is: it is not among the bytes that move
    every = 2 * sum(v.nbytes for v in st_h.values()) + sum(v.nbytes for v in out_h.values())
    assert pinned != "all" or moved[0] < every - st_h["act_id"].nbytes + (0 if probs is None else probs.nbytes)
    r.close()


class _HostStep:
    """Host-buffer steps on buffers that `place` makes from pageable ones."""

    def __init__(self, cfg, wl, place, fscore):
        n = wl.state["step"].shape[0]
        self.r, self.best = Router(wl, device="cuda:0"), 1e30
        self.st = {k: place(v.cpu()) for k, v in self.r.device_state().items()}
        self.out = {k: place(v) for k, v in self.r.outputs(n, device="cpu", fscore=fscore).items()}
        self.probs = place(torch.full((n, cfg.G, cfg.B, cfg.H), 0.02)) if cfg.H else None

    def step(self):
        t0 = time.perf_counter()
        self.r.step_host(self.st, self.out, self.probs)
        self.best = min(self.best, time.perf_counter() - t0)


def _faster(cfg, wl, place, other, factor, fscore):
    """Whether the shortest step with `place` takes less than `factor` times the shortest with `other`.  The bus has other
    users, and for seconds at a time every step takes up to twice as long, so the two are timed in turn, and over
    more rounds while the answer is no: a difference that is there stays in the shortest of them."""
    a, b = _HostStep(cfg, wl, place, fscore), _HostStep(cfg, wl, other, fscore)
    for _ in range(8):
        for _ in range(12):
            a.step()
            b.step()
        if a.best < factor * b.best:
            break
        time.sleep(0.2)
    a.r.close()
    b.r.close()
    return a.best < factor * b.best


def _page_locked_off_16(t):
    buf = torch.empty(t.numel() * t.element_size() + 8, dtype=torch.uint8).pin_memory()
    w = buf[8:].view(t.dtype).view(t.shape)
    w.copy_(t)
    return w


def test_score_matrix_is_not_slower_page_locked():
    # written an element at a time (in place it took 2.4 times as long as from pageable memory)
    cfg = wlm.get_config("c3")
    wl = wlm.make_workload(cfg, n_instances=512)
    assert _faster(cfg, wl, torch.Tensor.pin_memory, lambda t: t.clone(), 1.0, True)


def test_terminations_from_classifier_rows_are_not_slower_in_place():
    # every row is read: 1.35 times as long in place at this size as from arrays that no kernel can use in place; both
    # are copied now, and a fifth is left for the bus's other users
    cfg = wlm.get_config("c4", term_mode=2, burst_every=0, init_active=60)
    wl = wlm.make_workload(cfg, n_instances=63)
    assert _faster(cfg, wl, torch.Tensor.pin_memory, _page_locked_off_16, 1.2, False)


@pytest.mark.parametrize("name,n_inst", [("c3", 3), ("c3", 520), ("c2", 3)])
def test_score_matrix_to_page_locked_memory(name, n_inst):
    cfg = wlm.get_config(name)
    wl = wlm.make_workload(cfg, n_instances=n_inst)
    r = Router(wl, device="cuda:0")
    st_d, out_d = r.device_state(), r.outputs(n_inst, fscore=True)
    st_h = {k: v.cpu().pin_memory() for k, v in st_d.items()}
    out_h = {k: v.cpu().pin_memory() for k, v in out_d.items()}
    probs = torch.from_numpy(np.ascontiguousarray(wlm.term_probs_np(wl, 0))) if cfg.H else None
    r.step_host(st_h, out_h, None if probs is None else probs.pin_memory())
    r.step(st_d, out_d, None if probs is None else probs.cuda())
    for a, b in ((out_h, out_d), (st_h, st_d)):
        for key in a:
            assert torch.equal(a[key], b[key].cpu()), key
    r.close()
