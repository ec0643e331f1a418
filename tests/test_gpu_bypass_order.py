"""br_bypass_dispatch may become resident while the kernel ahead of it still runs: what that kernel writes is what it reads, in
eager streams and in captured graphs.  Whole numbers against the oracle: the tolerance is equality."""
import numpy as np
import pytest
import torch

import oracle
from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import Router

pytestmark = pytest.mark.gpu


def _check(G, s, L, infl, cap, got):
    for n in range(len(s)):
        want, Lw, nw = oracle.bypass(G, s[n], L[n], infl[n], cap[n], score_mode=0, alpha=1.0, beta=float(G))
        assert np.array_equal(got[0][n], want), n
        assert np.array_equal(got[1][n], Lw) and np.array_equal(got[2][n], nw), n


def _router(G):
    return Router(wlm.make_workload(wlm.get_config("c3", G=G, init_active=8, init_queue=0), n_instances=1), device="cuda:0")


def _inputs(G, N, n_req):
    gen = torch.Generator(device="cuda").manual_seed(G + n_req)
    s = torch.randint(1, 30000, (N, n_req), generator=gen, device="cuda", dtype=torch.int32)
    L = torch.randint(0, 400000, (N, G), generator=gen, device="cuda", dtype=torch.int64)
    infl = torch.randint(0, 3, (N, G), generator=gen, device="cuda", dtype=torch.int32)
    cap = torch.randint(1, 3 + 2 * n_req // G, (N, G), generator=gen, device="cuda", dtype=torch.int32)
    return s, L, infl, cap


@pytest.mark.parametrize("G,N,n_req", [(32, 1, 200), (33, 300, 33), (7, 2000, 64)])
def test_inputs_written_by_the_kernel_ahead(G, N, n_req):
    r = _router(G)
    s, L, infl, cap = _inputs(G, N, n_req)
    rounds = 25
    lens, loads, runs = torch.empty_like(s), torch.empty_like(L), torch.empty_like(infl)
    out = torch.empty((rounds, N, n_req), dtype=torch.int32, device="cuda")
    kept = []
    torch.cuda.synchronize()
    for k in range(rounds):                               # nothing waits for the host in between
        torch.mul(L, k + 1, out=loads)
        torch.add(infl, k % 3, out=runs)
        torch.add(s, 17 * k, out=lens)                    # the kernel directly ahead
        r.bypass_dispatch(lens, loads, runs, cap, out[k])
        if k in (0, 11, rounds - 1):
            kept.append((k, loads.clone(), runs.clone()))
    torch.cuda.synchronize()
    sn, Ln, fn, cn = (x.cpu().numpy() for x in (s, L, infl, cap))
    for k, lo, ru in kept:
        _check(G, sn + np.int32(17 * k), Ln * (k + 1), fn + np.int32(k % 3), cn, (out[k].cpu().numpy(), lo.cpu().numpy(), ru.cpu().numpy()))
    r.close()


@pytest.mark.parametrize("G,N,n_req", [(32, 400, 20), (64, 3000, 33)])
def test_dispatches_that_share_their_loads(G, N, n_req):
    r = _router(G)
    s, L, infl, cap = _inputs(G, N, 4 * n_req)
    parts = [p.contiguous() for p in s.split(n_req, dim=1)]
    out = torch.empty((len(parts), N, n_req), dtype=torch.int32, device="cuda")
    loads, runs = L.clone(), infl.clone()
    torch.cuda.synchronize()
    for p, o in zip(parts, out):
        r.bypass_dispatch(p, loads, runs, cap, o)
    torch.cuda.synchronize()
    got = torch.cat(list(out), dim=1).cpu().numpy()
    _check(G, *(x.cpu().numpy() for x in (s, L, infl, cap)), (got, loads.cpu().numpy(), runs.cpu().numpy()))
    r.close()


@pytest.mark.parametrize("ahead", ["copy", "kernel", "dispatch"])
def test_captured_by_the_caller(ahead):
    G, N, n_req = 32, 200, 40
    r = _router(G)
    s, L, infl, cap = _inputs(G, N, n_req)
    lens, loads, runs = s.clone(), torch.empty_like(L), torch.empty_like(infl)
    out = torch.empty((N, n_req), dtype=torch.int32, device="cuda")

    def tick():
        loads.copy_(L)
        runs.copy_(infl)
        if ahead == "kernel":
            torch.add(s, 5, out=lens)
        if ahead == "dispatch":
            r.bypass_dispatch(lens, loads, runs, cap, out)
        r.bypass_dispatch(lens, loads, runs, cap, out)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        tick()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        tick()
    for k in range(3):
        s += 3
        L += 1000 * k
        if ahead != "kernel":
            lens.copy_(s)
        graph.replay()
        torch.cuda.synchronize()
        sn, Ln, fn, cn = (x.cpu().numpy() for x in (lens, L, infl, cap))
        if ahead == "dispatch":
            first = [oracle.bypass(G, sn[n], Ln[n], fn[n], cn[n], score_mode=0, alpha=1.0, beta=float(G)) for n in range(N)]
            Ln, fn = np.stack([f[1] for f in first]), np.stack([f[2] for f in first])
        _check(G, sn, Ln, fn, cn, (out.cpu().numpy(), loads.cpu().numpy(), runs.cpu().numpy()))
    r.close()
