"""The routing step at the sizes its users run it at, through the calls of
``paper_2605_06113_b200.binding.Router``.

Five kinds of call:

* ``tick``   one cluster, one decode step per call, the latency path of a live dispatcher (a replayed
             graph, or an eager ``step`` where the caller's buffers change from call to call);
* ``batch``  many independent clusters on device buffers, one or several decode steps per call
             (simulation, parameter studies, replays);
* ``host``   the stateless step: the whole snapshot in pinned host buffers, up and down on every call;
* ``fscore`` the F-score matrix with the best worker per request;
* ``bypass`` pool-bypass dispatch of a tick's new requests on virtual loads.

Shapes, length distributions, arrival rates and router parameters are those of the configurations
in ``workload.py`` (c0, c1, c3, c4, h80) and of the ragged shapes of the tests.  Clusters start close
to saturation (a few percent of the slots free, the queue full), which is where the router works; they
then evolve by their own arrivals and terminations, so repeated passes walk a stationary regime.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2605_06113_b200 import workload as wlm
from paper_2605_06113_b200.binding import EMPTY, Router

DEVICE = "cuda:0"
TAB = 1 << wlm.TAB_LOG2

# term: "hazard" (every slot ends with probability 1 / mean_out per step), "classifier" (Bernoulli of the
# classifier's first probability), "lifetime" (requests carry their output length; perfect-lookahead c_hat)
_STEP = dict(N=1, G=16, B=64, W=512, H=0, R_max=4, n_steps=1, graph=False, term="hazard", mean_out=500.0,
             rate_lo=8.0, rate_hi=8.0, burst=0, mu=7.0, sigma=1.0, gate=0.5, fill=0.97, queue=1.0)


def _case(kind, name, **kw):
    base = dict(_STEP) if kind in ("tick", "batch", "host") else {}
    base.update(kw, kind=kind, name=name)
    return base


def listed():
    return [
        # the smallest fleet, stepped eagerly: launch and call overhead
        _case("tick", "tick_br0_g4", G=4, W=128, rate_lo=2.0, rate_hi=2.0),
        # a live BR-0 dispatcher, 16 workers and a queue of 512
        _case("tick", "tick_br0_g16", G=16, W=512, mean_out=400.0, graph=True),
        # a live BR-H dispatcher at the largest fleet: 64 workers, 1,024 waiting, classifier-driven c_hat
        _case("tick", "tick_brh_g64_h8", G=64, W=1024, H=8, mean_out=600.0, rate_lo=20.0, rate_hi=20.0,
              burst=200, mu=8.0, sigma=1.5, graph=True),
        # the deployed lookahead, H = 80, on 8 workers
        _case("tick", "tick_brh_g8_h80", G=8, W=512, H=80, term="lifetime", rate_lo=0.7, rate_hi=0.7, mu=8.0,
              sigma=0.8, fill=0.97, queue=0.5, graph=True),
        # throughput of BR-0 over 4,096 clusters: a step per call, and a stretch of steps per call
        _case("batch", "batch_br0_step", N=4096, G=32, W=256, rate_lo=4.0, rate_hi=16.0, mu=7.5, sigma=1.2),
        _case("batch", "batch_br0_run16", N=4096, G=32, W=256, rate_lo=4.0, rate_hi=16.0, mu=7.5, sigma=1.2,
              n_steps=16),
        # throughput of BR-H over 1,024 large clusters, new classifier output every step
        _case("batch", "batch_brh_step", N=1024, G=64, W=1024, H=8, mean_out=600.0, rate_lo=20.0, rate_hi=20.0,
              burst=200, mu=8.0, sigma=1.5),
        # odd sizes throughout, terminations drawn from the classifier's own output, three steps per call
        _case("batch", "batch_brh_ragged", N=777, G=21, B=40, W=300, H=6, R_max=5, term="classifier", gate=0.1,
              rate_lo=20.0, rate_hi=40.0, n_steps=3),
        # the deployed lookahead over 1,024 clusters, eight steps per call
        _case("batch", "batch_brh_h80_run8", N=1024, G=8, W=512, H=80, term="lifetime", rate_lo=0.7, rate_hi=0.7,
              mu=8.0, sigma=0.8, queue=0.5, n_steps=8),
        # the stateless step from and to host memory
        _case("host", "host_br0", N=4096, G=32, W=256, rate_lo=4.0, rate_hi=16.0, mu=7.5, sigma=1.2),
        # the score matrix of Eq. 2 for 200 snapshots
        _case("fscore", "fscore_h8", N=200, n=1024, G=64, H=8, mu=8.0, sigma=1.5),
        # pool bypass: 256 clusters dispatch a tick's 200 arrivals each
        _case("bypass", "bypass_g32", N=256, n=200, G=32, mu=7.5, sigma=1.2),
    ]


# ----------------------------------------------------------------------------- drawn cases
def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _weight(c):
    w = work(c)
    return max(w["bytes"], w["flops"] / 50.0)


def draw(rng):
    kind = rng.choice(["tick", "tick", "batch", "batch", "batch", "host", "fscore", "bypass"])
    most = max(_weight(c) for c in listed() if c["kind"] == kind)
    mu, sigma = rng.uniform(6.5, 8.0), rng.uniform(0.8, 1.5)
    if kind in ("fscore", "bypass"):
        c = dict(kind=kind, N=_log(rng, 1, 512), n=4 * _log(rng, 2, 512), G=_log(rng, 2, 64),
                 H=rng.choice([0, rng.randint(1, 16)]) if kind == "fscore" else 0, mu=mu, sigma=sigma)
    else:
        router = "br0" if kind == "host" else rng.choice(["br0", "classifier", "lifetime"])
        G, B = _log(rng, 2, 64), 8 * rng.choice([3, 5, 8, 8, 8, 12])
        c = dict(_STEP, kind=kind, G=G, B=B, W=4 * _log(rng, 8, 256), R_max=rng.choice([2, 4, 4, 5]),
                 mu=mu, sigma=sigma, fill=rng.uniform(0.8, 0.99), queue=rng.uniform(0.3, 1.0))
        c["N"] = 1 if kind == "tick" else _log(rng, 16 if kind == "host" else 48, 4096)
        c["n_steps"] = 1 if kind == "host" else rng.choice([1, 1, rng.randint(2, 16)])
        c["graph"] = kind == "tick" and rng.random() < 0.5
        c["mean_out"] = rng.uniform(200.0, 800.0)
        if router == "classifier":
            c["H"], c["gate"] = rng.randint(1, 16), rng.choice([0.1, 0.5])
            c["term"] = rng.choice(["hazard", "classifier"])
        elif router == "lifetime":
            c["H"], c["term"] = rng.randint(12, 80), "lifetime"
        ends = G * B / (26.0 if c["term"] == "classifier" else 1100.0 if c["term"] == "lifetime" else c["mean_out"])
        c["rate_lo"] = min(24.0, max(0.3, ends * rng.uniform(0.8, 1.3)))     # near saturation
        c["rate_hi"] = min(32.0, c["rate_lo"] * rng.uniform(1.0, 2.0))
    while _weight(c) > most and c["N"] > 1:
        c["N"] = max(1, c["N"] * 3 // 4)
    while _weight(c) > most and c.get("n_steps", 1) > 1:
        c["n_steps"] -= 1
    return c


# ----------------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=None)
def _lengths(mu, sigma, lo, hi):
    return wlm.lognormal_table(mu, sigma, lo, hi)


@functools.lru_cache(maxsize=None)
def _beta(a, b):
    return wlm.beta_table(a, b)


@functools.lru_cache(maxsize=None)
def _poisson(lo, hi):
    return wlm.poisson_thresholds(np.linspace(lo, hi, 64))


@functools.lru_cache(maxsize=None)
def _on_device(fn, *args):
    return torch.from_numpy(fn(*args)).to(DEVICE)


def _config(c):
    term = dict(hazard=1, classifier=2, lifetime=3)[c["term"]]
    kw = dict(beta=48.0, gamma=0.9, pred_mode=1) if term == 3 else {}
    return wlm.Config("case", N=c["N"], G=c["G"], W=c["W"], H=c["H"], steps=1, first_seed=0, init_active=0,
                      init_queue=0, len_mu=c["mu"], len_sigma=c["sigma"], arrival=("const", 1.0),
                      hazard=1.0 / c["mean_out"] if term == 1 else 0.0, term_mode=term, B=c["B"], R_max=c["R_max"],
                      gate=c["gate"], beta_ab=(2.0, 50.0) if term == 2 else (2.0, 60.0),
                      burst_every=250 if c["burst"] else 0, burst_size=c["burst"],
                      ctx_clip=(16, 131072), **kw).resolved()


def _draws(gen, table, *shape):
    """table values at uniformly drawn indexes"""
    return table[torch.randint(TAB, shape, generator=gen, device=DEVICE)]


def _step_state(c, seed):
    cfg, N, G, B, W, H = _config(c), c["N"], c["G"], c["B"], c["W"], c["H"]
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    i32 = torch.int32
    s_tab = _on_device(_lengths, c["mu"], c["sigma"], 1, 131072)
    cur = _draws(gen, _on_device(_lengths, c["mu"], c["sigma"], 16, 131072), N, G, B)
    run = torch.rand((N, G, B), generator=gen, device=DEVICE) < c["fill"]
    words = (B + 63) // 64
    bits = torch.zeros((N, G, words * 64), dtype=torch.int64, device=DEVICE)
    bits[:, :, :B] = run
    occ = (bits.view(N, G, words, 64) << torch.arange(64, device=DEVICE)).sum(-1)
    slot = torch.arange(G * B, dtype=i32, device=DEVICE).view(1, G, B)
    n_q = int(W * c["queue"])
    waiting = torch.arange(W, device=DEVICE) < n_q
    st = dict(load=torch.where(run, cur, 0).sum(2, dtype=torch.int64), nact=run.sum(2, dtype=i32), occ=occ,
              act_base=torch.where(run, cur, EMPTY), act_id=torch.where(run, slot, -1),
              step=torch.zeros(N, dtype=i32, device=DEVICE),
              seed=torch.randint(1 << 40, (N,), generator=gen, device=DEVICE),
              next_id=torch.full((N,), G * B + n_q, dtype=i32, device=DEVICE),
              wq_s=torch.where(waiting, _draws(gen, s_tab, N, W), 0),
              wq_id=torch.where(waiting, G * B + torch.arange(W, dtype=i32, device=DEVICE), 0).repeat(N, 1),
              wq_n=torch.full((N,), n_q, dtype=i32, device=DEVICE))
    probs, out_tab = [], None
    if c["term"] == "lifetime":
        out_tab = _lengths(cfg.out_mu, cfg.out_sigma, *cfg.out_clip)
        o_tab = _on_device(_lengths, cfg.out_mu, cfg.out_sigma, *cfg.out_clip)
        left = _draws(gen, o_tab, N, G, B) * torch.rand((N, G, B), generator=gen, device=DEVICE)
        st.update(act_end=torch.where(run, left.to(i32), 0), wq_o=torch.where(waiting, _draws(gen, o_tab, N, W), 0))
    elif H:
        age = torch.randint(cfg.delta_T, (N, G, B), generator=gen, device=DEVICE)
        st.update(act_chat0=torch.full((N, G, B), float(H), device=DEVICE), act_kref=(-age & 255).to(torch.uint8))
        # one block of classifier output per decode step, two calls' worth (a replayed graph reads one block)
        for _ in range(1 if c["graph"] else 2):
            probs.append(_draws(gen, _on_device(_beta, *cfg.beta_ab), c["n_steps"], N, G, B, H))
    rates = _poisson(c["rate_lo"], c["rate_hi"])[np.random.default_rng(seed).integers(64, size=N)]
    wl = wlm.Workload(cfg=cfg, seeds=np.zeros(N, np.uint64), len_tab=_lengths(c["mu"], c["sigma"], 1, 131072),
                      beta_tab=None, arr_cdf=rates, arr_period=1, arr_inst_stride=1,
                      term_cdf=wlm.termination_gap_thresholds(cfg.hazard, B), out_tab=out_tab)
    return wl, st, probs


def prepare(case, seed):
    c = case
    if c["kind"] in ("tick", "batch", "host"):
        wl, st, probs = _step_state(c, seed)
        r = Router(wl, device=DEVICE)
        if c["kind"] == "host":
            st = {k: v.cpu().pin_memory() for k, v in st.items()}
            out = {k: v.pin_memory() for k, v in r.outputs(c["N"], device="cpu").items()}
        else:
            out = r.outputs(c["N"], n_steps=c["n_steps"])
        if c["graph"]:
            r.graph_capture(st, out, probs[0] if probs else None, n_steps=c["n_steps"])
        return dict(case=c, router=r, st=st, out=out, probs=probs, calls=0)

    N, n, G, H = c["N"], c["n"], c["G"], c["H"] if c["kind"] == "fscore" else 0
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    cfg = wlm.Config("case", N=N, G=G, W=256, H=H, steps=1, first_seed=0, init_active=0, init_queue=0,
                     len_mu=c["mu"], len_sigma=c["sigma"], arrival=("const", 1.0), hazard=0.002).resolved()
    wl = wlm.Workload(cfg=cfg, seeds=np.zeros(N, np.uint64), len_tab=_lengths(c["mu"], c["sigma"], 1, 131072),
                      beta_tab=None, arr_cdf=_poisson(1.0, 1.0), arr_period=1, arr_inst_stride=0,
                      term_cdf=wlm.termination_gap_thresholds(cfg.hazard, cfg.B))
    r = Router(wl, device=DEVICE)
    s_tab = _on_device(_lengths, c["mu"], c["sigma"], 1, 131072)
    s = _draws(gen, s_tab, N, n)
    load = _draws(gen, s_tab, N, G, 60).sum(2, dtype=torch.int64)            # about 60 running requests a worker
    st = dict(case=c, router=r, s=s)
    if c["kind"] == "fscore":
        # projected loads: a few requests leave at every offset, the others grow by a token
        leave = _draws(gen, s_tab, N, G, H + 1).to(torch.int64) * (torch.rand((N, G, H + 1), generator=gen, device=DEVICE) < 0.3)
        leave[:, :, 0] = 0
        grow = 60 * torch.arange(H + 1, device=DEVICE)
        st.update(Lh=(load[:, :, None] - leave.cumsum(2)).clamp_(min=0) + grow,
                  cap=torch.randint(0, 4, (N, G), generator=gen, device=DEVICE, dtype=torch.int32),
                  F=torch.empty((N, n, G), dtype=torch.float64, device=DEVICE),
                  best=torch.empty((N, n), dtype=torch.int32, device=DEVICE))
    else:
        # the engines' last report; caps leave room for most of a tick's arrivals
        st.update(reported=load, running=torch.randint(40, 64, (N, G), generator=gen, device=DEVICE, dtype=torch.int32),
                  cap=torch.randint(64, 64 + max(2, 2 * n // G), (N, G), generator=gen, device=DEVICE, dtype=torch.int32),
                  vload=torch.empty_like(load), inflight=torch.empty((N, G), dtype=torch.int32, device=DEVICE),
                  worker=torch.empty((N, n), dtype=torch.int32, device=DEVICE))
    return st


# ----------------------------------------------------------------------------- one pass
def run(state):
    c, r = state["case"], state["router"]
    if c["kind"] == "fscore":
        r.fscore(state["s"], state["Lh"], state["F"], cap=state["cap"], best_g=state["best"])
        return state["F"], state["best"]
    if c["kind"] == "bypass":
        # every tick starts from the engines' report
        state["vload"].copy_(state["reported"])
        state["inflight"].copy_(state["running"])
        r.bypass_dispatch(state["s"], state["vload"], state["inflight"], state["cap"], state["worker"])
        return state["worker"], state["vload"], state["inflight"]
    st, out = state["st"], state["out"]
    if c["kind"] == "host":
        r.step_host(st, out)
    elif c["graph"]:
        r.graph_step()
    else:
        probs = state["probs"]
        r.step(st, out, probs[state["calls"] % len(probs)] if probs else None, n_steps=c["n_steps"])
        state["calls"] += 1
    return out, st


# ----------------------------------------------------------------------------- what a pass cannot do without
def _per_step(c):
    """(running-request terms, bytes, admissions, score evaluations) of one instance and decode step"""
    G, W, H, A = c["G"], c["W"], c["H"], c["G"] * c["B"]
    life = c["term"] == "lifetime"
    ends = A / (26.0 if c["term"] == "classifier" else 1100.0 if life else c["mean_out"])
    adm = min(ends, 0.5 * (c["rate_lo"] + c["rate_hi"]))
    # running lengths and queue in, assignments out, per-worker state in and out, slots edited
    b = 4.0 * A + 8.0 * W + 4.0 * W + 48.0 * G + 24.0 + 16.0 * (adm + ends)
    if life:
        b += 4.0 * A + 8.0 * W                                   # the step each request ends at, output lengths
    elif H:
        period = max(1, H // 2)
        b += 4.0 * A + 4.0 * A / period                          # c_hat in, refreshed ones out
        b += 4.0 * H * A * (1.0 if c["term"] == "classifier" else 1.0 / period)
    flops = adm * (2 ** c["R_max"] - 1 + W) * (4.0 * (H + 1) + 3.0) + 2.0 * A
    return b, flops


def work(case):
    c = case
    if c["kind"] == "fscore":
        scores = float(c["N"]) * c["n"] * c["G"]
        return {"bytes": 8.0 * scores + c["N"] * (8.0 * c["n"] + c["G"] * (8.0 * (c["H"] + 1) + 4.0)),
                "flops": scores * (4.0 * (c["H"] + 1) + 3.0)}
    if c["kind"] == "bypass":
        return {"bytes": c["N"] * (8.0 * c["n"] + 40.0 * c["G"]), "flops": 6.0 * c["N"] * c["n"] * c["G"]}
    b, f = _per_step(c)
    return {"bytes": b * c["N"] * c["n_steps"], "flops": f * c["N"] * c["n_steps"]}


def tolerance(case):
    # assignments, loads and every array of the snapshot are whole numbers; the fp64 scores and the fp32
    # c_hat are evaluated term by term in the order that the definitions state, so they are equal too
    return "exact"
