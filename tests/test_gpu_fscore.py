"""br_fscore (the F-score matrix and the pool-bypass arg-max) against the checker's Eq. 1 / Eq. 2."""
import ctypes as C

import numpy as np
import pytest
import torch

import oracle
from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,H", [("c3", 0), ("c4", 8), ("c2", 4), ("h80", 80), ("c4", 33)])
def test_fscore_matrix_and_best_worker(name, H):
    cfg = wlm.get_config(name, H=H)
    wl = wlm.make_workload(cfg, n_instances=2)
    r = Router(wl, device="cuda:0")
    rng = np.random.default_rng(3 + H)
    N, G, n_req = 3, cfg.G, 2052                      # two full tiles and a ragged tail
    s = rng.integers(1, 60000, (N, n_req)).astype(np.int32)
    Lh = rng.integers(100000, 400000, (N, G, H + 1)).astype(np.int64)
    cap = rng.integers(0, 3, (N, G)).astype(np.int32)
    cap[2] = 0                                        # no worker has room: best_g = -1
    st, Lt, ct = (torch.from_numpy(x).cuda() for x in (s, Lh, cap))
    F = torch.zeros((N, n_req, G), dtype=torch.float64, device="cuda")
    best = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.fscore(st, Lt, F, cap=ct, best_g=best)
    torch.cuda.synchronize()
    Fh, bh = F.cpu().numpy(), best.cpu().numpy()
    M = Lh.max(axis=1)                                # envelope per offset
    for n in range(N):
        for i in list(range(0, 40)) + list(range(n_req - 40, n_req)) + [int(x) for x in rng.integers(0, n_req, 60)]:
            ref = np.empty(G)
            for g in range(G):
                m = M[n] - Lh[n, g]
                if cfg.score_mode == 0:
                    ref[g] = oracle.f_br0(G, int(s[n, i]), int(m[0]))
                else:
                    ref[g] = oracle.f_brh(H, cfg.alpha, cfg.beta, cfg.gamma, int(s[n, i]), m)
            err = np.abs(Fh[n, i] - ref) / np.maximum(1.0, np.abs(ref))
            assert err.max() <= 1e-6                  # stated tolerance
            assert np.array_equal(Fh[n, i], ref)      # same arithmetic, same order: equality
            ok = np.nonzero(cap[n] > 0)[0]
            want = -1 if len(ok) == 0 else int(ok[np.argmax(ref[ok])])
            assert bh[n, i] == want
    r.close()


@pytest.mark.parametrize("G", [1, 2, 7, 9, 33, 64])
@pytest.mark.parametrize("H", [0, 3, 4, 18])
@pytest.mark.parametrize("n_req", [4, 60, 64, 260])
def test_fscore_edges(G, H, n_req):
    # requests at a worker's smallest margin and one token on either side of it, loads beyond 32 bits (the order of
    # the terms and every rounding is the checker's: equality)
    cfg = wlm.get_config("c2", G=G, H=H, init_active=2, init_queue=0, term_mode=1, score_mode=1)
    r = Router(wlm.make_workload(cfg, n_instances=1), device="cuda:0")
    rng = np.random.default_rng(G + 100 * H + n_req)
    N = 3
    Lh = rng.integers(1000, 9000, (N, G, H + 1)).astype(np.int64)
    Lh[1] += np.int64(1) << 40
    Lh[2, G - 1] += np.int64(1) << 34
    mm = (Lh.max(axis=1, keepdims=True) - Lh).min(axis=2)
    s = np.clip(mm[:, rng.integers(0, G, n_req)] + rng.integers(-1, 2, (N, n_req)), 1, 200000).astype(np.int32)
    s[:, 0] = 1
    st, Lt = torch.from_numpy(s).cuda(), torch.from_numpy(Lh).cuda()
    F = torch.zeros((N, n_req, G), dtype=torch.float64, device="cuda")
    best = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.fscore(st, Lt, F, best_g=best)
    Fh, bh = F.cpu().numpy(), best.cpu().numpy()
    for n in range(N):
        M = Lh[n].max(axis=0)
        for i in list(range(0, n_req, 7)) + [n_req - 1]:
            ref = np.array([oracle.f_brh(H, cfg.alpha, cfg.beta, cfg.gamma, int(s[n, i]), M - Lh[n, g]) for g in range(G)])
            assert np.array_equal(Fh[n, i], ref), (n, i)
            assert bh[n, i] == int(np.argmax(ref)), (n, i)
    r.close()


@pytest.mark.parametrize("G", [1, 2, 7, 9, 31, 33, 64])
@pytest.mark.parametrize("N,n_req", [(1, 4), (3, 60), (3, 64), (2, 260), (40, 1100)])
@pytest.mark.parametrize("with_cap", [False, True])
def test_fscore_edges_in_integers(G, N, n_req, with_cap):
    # Eq. 1: the walk over (request, worker) at every remainder of 32 by G, warps with 64 requests and with fewer, and the
    # best worker among all and among those with room
    cfg = wlm.get_config("c3", G=G, init_active=2, init_queue=0)
    assert cfg.score_mode == 0
    r = Router(wlm.make_workload(cfg, n_instances=1), device="cuda:0")
    rng = np.random.default_rng(G + 7 * n_req)
    Lh = rng.integers(1000, 9000, (N, G, 1)).astype(np.int64)
    if N > 1:
        Lh[1] += np.int64(1) << 40
    m = Lh.max(axis=1, keepdims=True) - Lh
    s = np.clip(m[:, rng.integers(0, G, n_req), 0] + rng.integers(-1, 2, (N, n_req)), 1, 200000).astype(np.int32)
    cap = rng.integers(0, 2, (N, G)).astype(np.int32)
    cap[0] = 0
    st, Lt, ct = (torch.from_numpy(x).cuda() for x in (s, Lh, cap))
    F = torch.zeros((N, n_req, G), dtype=torch.float64, device="cuda")
    best = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.fscore(st, Lt, F, cap=ct if with_cap else None, best_g=best)
    ref = np.array([[[oracle.f_br0(G, int(x), int(y)) for y in m[n, :, 0]] for x in s[n]] for n in range(min(N, 3))], dtype=np.float64)
    over = np.maximum(s[:, :, None].astype(np.int64) - m[:, None, :, 0], 0)
    every = (s[:, :, None].astype(np.int64) - G * over).astype(np.float64)
    assert np.array_equal(ref, every[:3])
    assert np.array_equal(F.cpu().numpy(), every)
    room = cap > 0 if with_cap else np.ones((N, G), dtype=bool)
    masked = np.where(room[:, None, :], every, -np.inf)
    assert np.array_equal(best.cpu().numpy(), np.where(room.any(axis=1)[:, None], masked.argmax(axis=2), -1))
    r.close()


@pytest.mark.parametrize("G", [1, 2, 3, 17, 32, 33])
@pytest.mark.parametrize("H", [31, 78, 80])
def test_fscore_long_horizons_on_small_fleets(G, H):
    # margins taken four offsets at a time, of which the last warp's may be fewer; equality
    cfg = wlm.get_config("h80", G=G, H=H, init_active=2, init_queue=0)
    r = Router(wlm.make_workload(cfg, n_instances=1), device="cuda:0")
    rng = np.random.default_rng(G + H)
    N, n_req = 2, 12
    Lh = rng.integers(1000, 9000, (N, G, H + 1)).astype(np.int64)
    s = rng.integers(1, 9000, (N, n_req)).astype(np.int32)
    st, Lt = torch.from_numpy(s).cuda(), torch.from_numpy(Lh).cuda()
    F = torch.zeros((N, n_req, G), dtype=torch.float64, device="cuda")
    best = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.fscore(st, Lt, F, best_g=best)
    Fh, bh = F.cpu().numpy(), best.cpu().numpy()
    for n in range(N):
        M = Lh[n].max(axis=0)
        for i in range(n_req):
            ref = np.array([oracle.f_brh(H, cfg.alpha, cfg.beta, cfg.gamma, int(s[n, i]), M - Lh[n, g]) for g in range(G)])
            assert np.array_equal(Fh[n, i], ref) and bh[n, i] == int(np.argmax(ref)), (n, i)
    r.close()


@pytest.mark.parametrize("G,score_mode", [(32, 0), (64, 0), (5, 0), (16, 1)])
def test_pool_bypass_dispatch(G, score_mode):
    """br_bypass_dispatch against the checker: workers, virtual loads and inflight counts."""
    kw = dict(G=G, init_active=8, init_queue=0)
    if score_mode == 1:
        kw.update(score_mode=1, alpha=1.0, beta=7.5, gamma=1.0)
    cfg = wlm.get_config("c3", **kw)
    wl = wlm.make_workload(cfg, n_instances=1)
    r = Router(wl, device="cuda:0")
    rng = np.random.default_rng(71 + G)
    N, n_req = 9, 150
    s = rng.integers(1, 40000, (N, n_req)).astype(np.int32)
    s[0] = 1000                                            # equal lengths: ties between workers
    L = rng.integers(0, 300000, (N, G)).astype(np.int64)
    L[1] = 5000                                            # equal loads
    infl = rng.integers(0, 10, (N, G)).astype(np.int32)
    cap = rng.integers(8, 14, (N, G)).astype(np.int32)     # tight caps: some instances fill up
    cap[2] = 0
    st, Lt, it, ct = (torch.from_numpy(x.copy()).cuda() for x in (s, L, infl, cap))
    out = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.bypass_dispatch(st, Lt, it, ct, out)
    torch.cuda.synchronize()
    for n in range(N):
        want, Lw, nw = oracle.bypass(G, s[n], L[n], infl[n], cap[n], score_mode=score_mode, alpha=cfg.alpha,
                                     beta=float(G) if score_mode == 0 else cfg.beta)
        assert np.array_equal(out[n].cpu().numpy(), want), n
        assert np.array_equal(Lt[n].cpu().numpy(), Lw) and np.array_equal(it[n].cpu().numpy(), nw), n
    assert (out[2] == -1).all()
    r.close()


@pytest.mark.parametrize("G,n_req,lo,hi", [(1, 31, 1, 9), (2, 32, 1, 4), (33, 33, 1, 40000), (32, 1, 1, 9), (64, 97, 1 << 24, 1 << 26),
                                           (31, 64, (1 << 25) - 2, (1 << 25) + 2)])
def test_pool_bypass_edges(G, n_req, lo, hi):
    # whole and ragged groups of 32 requests, one and two workers per lane, lengths on either side of 2^25 (the packed
    # key's range), loads beyond 32 bits; whole numbers: equality
    cfg = wlm.get_config("c3", G=G, init_active=8, init_queue=0)
    r = Router(wlm.make_workload(cfg, n_instances=1), device="cuda:0")
    rng = np.random.default_rng(G + n_req)
    N = 5
    s = rng.integers(lo, hi, (N, n_req)).astype(np.int32)
    L = rng.integers(0, 3 * hi, (N, G)).astype(np.int64)
    L[0] = np.int64(1) << 40
    L[1, 0] = np.int64(1) << 40
    infl = rng.integers(0, 3, (N, G)).astype(np.int32)
    cap = rng.integers(0, 2 + 2 * n_req // G, (N, G)).astype(np.int32)
    st, Lt, it, ct = (torch.from_numpy(x.copy()).cuda() for x in (s, L, infl, cap))
    out = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.bypass_dispatch(st, Lt, it, ct, out)
    for n in range(N):
        want, Lw, nw = oracle.bypass(G, s[n], L[n], infl[n], cap[n], score_mode=0, alpha=1.0, beta=float(G))
        assert np.array_equal(out[n].cpu().numpy(), want), n
        assert np.array_equal(Lt[n].cpu().numpy(), Lw) and np.array_equal(it[n].cpu().numpy(), nw), n
    r.close()


@pytest.mark.parametrize("G", [31, 33, 64])
@pytest.mark.parametrize("n_req", [1, 45, 64])
def test_pool_bypass_scores_that_tie(G, n_req):
    # Eq. 2 scores with one and two workers per lane: equal virtual loads, among them those of workers g and g + 32, are
    # told apart by the lower index; the margins are re-based whenever the largest load grows.  Equality
    cfg = wlm.get_config("c3", G=G, init_active=8, init_queue=0, score_mode=1, alpha=1.0, beta=7.5, gamma=1.0)
    r = Router(wlm.make_workload(cfg, n_instances=1), device="cuda:0")
    rng = np.random.default_rng(G + n_req)
    N = 6
    s = rng.integers(1, 30000, (N, n_req)).astype(np.int32)
    s[0] = 700
    L = (rng.integers(0, 4, (N, G)) * 9000).astype(np.int64)               # many equal loads
    L[1] = 5000
    L[2, 32:] = L[2, :G - 32] if G > 32 else L[2, 32:]
    L[3] += np.int64(1) << 40
    infl = rng.integers(0, 3, (N, G)).astype(np.int32)
    cap = rng.integers(1, 4, (N, G)).astype(np.int32)
    cap[4, :G // 2] = 0
    st, Lt, it, ct = (torch.from_numpy(x.copy()).cuda() for x in (s, L, infl, cap))
    out = torch.full((N, n_req), -7, dtype=torch.int32, device="cuda")
    r.bypass_dispatch(st, Lt, it, ct, out)
    for n in range(N):
        want, Lw, nw = oracle.bypass(G, s[n], L[n], infl[n], cap[n], score_mode=1, alpha=cfg.alpha, beta=cfg.beta)
        assert np.array_equal(out[n].cpu().numpy(), want), n
        assert np.array_equal(Lt[n].cpu().numpy(), Lw) and np.array_equal(it[n].cpu().numpy(), nw), n
    r.close()



def test_empirical_survival_estimator():
    """br_survival_chat against the checker's counting definition (same fp64 operations: equality)."""
    cfg = wlm.get_config("c4")                              # H = 8
    wl = wlm.make_workload(cfg, n_instances=1)
    r = Router(wl, device="cuda:0")
    rng = np.random.default_rng(83)
    hist = np.sort(rng.geometric(1 / 600.0, 5000).astype(np.int32))
    prefix = np.concatenate([[0], np.cumsum(hist.astype(np.int64))]).astype(np.int64)
    age = np.concatenate([rng.integers(0, 3000, 3000), [0, int(hist[-1]) - 1, int(hist[-1]), int(hist[-1]) + 9,
                                                        int(hist[0]) - 1, int(hist[0])]]).astype(np.int32)
    ht, pt, at = (torch.from_numpy(x).cuda() for x in (hist, prefix, age))
    c = torch.empty(len(age), dtype=torch.float32, device="cuda")
    p = torch.empty(len(age), dtype=torch.float64, device="cuda")
    mu = torch.empty(len(age), dtype=torch.float64, device="cuda")
    r.survival_chat(ht, pt, at, c, p, mu)
    torch.cuda.synchronize()
    ch, ph, mh = c.cpu().numpy(), p.cpu().numpy(), mu.cpu().numpy()
    shuffled = rng.permutation(hist)                        # the definition does not need the order
    for i in list(range(400)) + list(range(len(age) - 6, len(age))):
        wc, wp, wm = oracle.survival(shuffled, cfg.H, int(age[i]))
        assert ch[i] == np.float32(wc) and ph[i] == wp and mh[i] == wm, i
    r.close()
