"""The calls a user of this library spends time in, as cases that can be timed.

Every case goes through the public binding (`paper_1402_2328_gb300`).  Kinds:

rounds  advance a replica-exchange Wang-Landau run by some rounds (`REWL.run`) and read the
        walkers' state back.  `stage` is -log2 of the ln f the windows are at: 0 is the opening
        of a cold start, 10..26 are the iterations a full run (1 -> 1e-8) spends its time in.
batch   the same for many uneven instances advanced together (`REWLBatch.run`).
start   `REWL.init`: seeded lattices, every walker driven into its window.
whole   a complete small run: init, rounds until done, joined ln g.
join    results of a finished run: joined ln g and its jackknife error.
em      production rounds with the (E, M) measurement, and the joint ln g(E, M).
thermo  canonical averages of a joined ln g.
train   Adam steps of the warm-start network.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1402_2328_gb300.rewl as R

OVERLAP = 0.75
# integer instructions one Wang-Landau attempt cannot do without (Philox4x32-10, site and
# neighbours, energy change, accept test, ln g / H update)
OPS_PER_ATTEMPT = 85


# ------------------------------------------------------------------------------- the cases
def _rounds(name, model, L, windows, walkers, stage, rounds, interval=10_000, flatness=0.8):
    return dict(name=name, kind="rounds", model=model, L=L, windows=windows, walkers=walkers,
                stage=stage, rounds=rounds, interval=interval, flatness=flatness)


def listed():
    return [
        # the smallest documented run (at most 250 of its rounds), from init to ln g: 4 walkers
        dict(name="whole_ising8", kind="whole", model=0, L=8, windows=4, walkers=1,
             lnf_final=1e-6, max_rounds=250),
        # few walkers on a middling lattice (the warm-start studies), middle iterations
        _rounds("ising32_mid", 0, 32, 8, 8, 12, 60),
        # Ising L=64, 32 x 16: the late iterations, where a run to 1e-8 spends its rounds
        _rounds("ising64_late", 0, 64, 32, 16, 20, 60),
        # q=10 Potts L=40, 64 x 16, middle iterations
        _rounds("potts40_mid", 10, 40, 64, 16, 10, 60),
        # q=10 Potts L=80, 64 x 16: opening rounds of a cold start (pre-runs, short studies);
        # a strict flatness keeps the run at ln f = 1
        _rounds("potts80_opening", 10, 80, 64, 16, 0, 60, flatness=0.95),
        # the same lattice in the last iterations: the longest runs of all
        _rounds("potts80_late", 10, 80, 64, 16, 24, 60),
        # 24 uneven instances advanced together: the largest number of walkers
        dict(name="batch24", kind="batch", instances=24, first=0, interval=10_000, rounds=12,
             stage=0),
        # starting the largest lattice: lattices seeded and 1024 walkers driven into their windows
        dict(name="start_potts80", kind="start", model=10, L=80, windows=64, walkers=16),
        # results of a finished Ising L=64 run
        dict(name="join_ising64", kind="join", model=0, L=64, windows=32, walkers=16),
        # production run of g(E, M) on the lattice size where the joint grid is still small
        dict(name="em_ising16", kind="em", L=16, windows=4, walkers=32, rounds=40),
        # u(T), c(T) curve of a joined ln g
        dict(name="thermo_ising64", kind="thermo", model=0, L=64, temperatures=500),
        # network of the learned warm start on its documented training set size: a few Adam steps
        dict(name="train_mlp", kind="train", samples=9716, steps=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bins(model, L):
    return L * L if model == 0 else 2 * L * L


def _draw_layout(rng, lmin, lmax, max_walkers=1024):
    """A lattice of either model with a window layout that the sampler can start."""
    model = rng.choice([0, 0, 10, 10, rng.randint(3, 9)])
    L = _log_int(rng, lmin, lmax)
    widest = max(2, min(64, _bins(model, L) // (12 * max(1, L // 8)) if model == 0 else
                        _bins(model, L) // 40))
    windows = min(widest, _log_int(rng, 2, 64))
    walkers = max(1, min(_log_int(rng, 1, 32), max_walkers // windows))
    return dict(model=model, L=L, windows=windows, walkers=walkers)


def draw(rng):
    kind = rng.choice(["rounds"] * 9 + ["batch"] * 2 + ["start", "whole", "join", "em", "thermo",
                                                        "train"])
    if kind == "rounds":
        interval = rng.choice([10_000, 10_000, _log_int(rng, 1000, 20_000)])
        return dict(kind=kind, **_draw_layout(rng, 8, 80), stage=rng.randint(0, 26),
                    rounds=max(2, int(rng.uniform(0.2, 1.0) * 600_000 / interval)),
                    interval=interval, flatness=rng.choice([0.8, 0.9, 0.95]))
    if kind == "batch":
        return dict(kind=kind, instances=rng.randint(2, 23), first=rng.randint(0, 40),
                    interval=_log_int(rng, 2000, 10_000), rounds=rng.randint(4, 12),
                    stage=rng.choice([0, rng.randint(1, 24)]))
    if kind == "start":
        return dict(kind=kind, **_draw_layout(rng, 8, 80))
    if kind == "whole":
        return dict(kind=kind, model=rng.choice([0, 3, 10]), L=rng.choice([4, 5, 6, 7, 8, 9, 10]),
                    windows=rng.randint(1, 2), walkers=rng.randint(1, 16),
                    lnf_final=10.0 ** -rng.uniform(2, 6), max_rounds=150)
    if kind == "join":
        return dict(kind=kind, **dict(_draw_layout(rng, 8, 64), walkers=rng.randint(2, 16)))
    if kind == "em":
        return dict(kind=kind, L=rng.choice([8, 10, 12, 13, 16]), windows=rng.randint(2, 4),
                    walkers=rng.randint(8, 32), rounds=rng.randint(10, 40))
    if kind == "thermo":
        return dict(kind=kind, model=rng.choice([0, 10, rng.randint(3, 9)]),
                    L=_log_int(rng, 6, 80), temperatures=_log_int(rng, 1, 500))
    return dict(kind=kind, samples=_log_int(rng, 100, 9716), steps=rng.randint(3, 12))


# ------------------------------------------------------------------------------- inputs
def _seed(seed, instance=0):
    return 0x5EED201400000000 + 1000 * (int(seed) % 1_000_000) + instance


def _zeros_like_state(r, field):
    return np.zeros_like(r.get_state(field))


def _move_to_stage(runner, handles, stage):
    """Runs a cold start down a short ladder of ln f values and leaves every window at
    ln f = 2^-stage, with an estimate of ln g like the one a run has by then."""
    if stage <= 0:
        runner.run(max_rounds=4)
        return
    runner.run(max_rounds=160)
    for e in (2, 4, 7, 11):
        if e < stage:
            for r in handles:
                r.set_state("lnf", np.full(r.h, 2.0 ** -e))
            runner.run(max_rounds=24)
    for r in handles:
        r.set_state("lnf", np.full(r.h, 2.0 ** -stage))
        r.set_state("iter", np.full(r.h, stage, np.int32))
        r.set_state("H", _zeros_like_state(r, "H"))
        r.set_state("flat", _zeros_like_state(r, "flat"))
    runner.run(max_rounds=2)


def _batch_descs(case, seed):
    """Ising L = 16, 32, 64 and q=10 Potts L = 20, 40 in turn, 8-64 windows, 4-16 walkers."""
    out = []
    for j in range(case["instances"]):
        i = case["first"] + j
        model, L = [(0, 16), (0, 32), (0, 64), (10, 20), (10, 40)][i % 5]
        out.append(dict(model=model, L=L, windows=[8, 16, 32, 64][i % 4],
                        walkers=[4, 8, 16][(i // 4) % 3], overlap=OVERLAP, lnf_final=1e-8,
                        flatness=0.8, seed=_seed(seed, j), instance=j))
    return out


def _finished(case, seed, interval=20_000, **params):
    """A run taken through all its iterations quickly: every check counts as flat."""
    r = R.REWL(case.get("model", 0), case["L"], case["windows"], OVERLAP, case["walkers"],
               2.0 ** -5, 0.0, seed=_seed(seed), interval=interval, **params)
    r.run(max_rounds=60)
    return r


def _smooth_lng(model, L):
    """A concave ln g over the bins with the ends and the area of a lattice's."""
    B, N, q = _bins(model, L), L * L, 2 if model == 0 else model
    k = np.arange(B + 1, dtype=np.float64)
    peak = B / 2.0 if model == 0 else 0.9 * B
    top = N * math.log(q)
    up = math.log(q) + (top - math.log(q)) * (1.0 - (1.0 - k / peak) ** 2)
    down = top - 0.5 * top * ((k - peak) / max(B - peak, 1.0)) ** 2
    lng = np.where(k <= peak, up, down)
    lng[[1, B - 1] if model == 0 else [1, 2, 3]] = -np.inf  # energies no lattice has
    return lng


def _thermo_inputs(case, seed):
    rng = np.random.default_rng(seed)
    lng = _smooth_lng(case["model"], case["L"])
    lng = lng + rng.normal(0.0, 0.05, lng.size)  # a run's statistical error
    T = np.sort(rng.uniform(0.4, 8.0, case["temperatures"]))
    return lng, T


def _train_inputs(case, seed):
    """Glorot weights; features (E/N, q, 1/L) and targets shaped like ln g / N."""
    rng = np.random.default_rng(seed)
    n = case["samples"]
    P = np.zeros(R.MLP_NPARAM, np.float32)
    for a, b, fan in ((0, 192, 67), (256, 4352, 128), (4416, 4480, 65)):
        P[a:b] = rng.uniform(-1.0, 1.0, b - a) * math.sqrt(6.0 / fan)
    e = rng.uniform(-2.0, 0.0, n)
    q = rng.choice([2.0, 10.0], n)
    il = 1.0 / rng.choice([8.0, 12.0, 16.0, 20.0, 24.0, 28.0, 32.0], n)
    X = np.stack([e, q, il], axis=1).astype(np.float32)
    T = (np.log(q) * (1 - (e / 2.0) ** 2) * (1 - 0.1 * il)).astype(np.float32)
    return P, X, T


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("rounds", "start"):
        r = R.REWL(case["model"], case["L"], case["windows"], OVERLAP, case["walkers"], 1e-8,
                   case.get("flatness", 0.8), seed=_seed(seed),
                   interval=case.get("interval", 10_000))
        if kind == "rounds":
            r.init()
            _move_to_stage(r, [r], case["stage"])
        return dict(case=case, r=r)
    if kind == "batch":
        b = R.REWLBatch(_batch_descs(case, seed), interval=case["interval"])
        b.init()
        handles = [b.instance(i) for i in range(case["instances"])]
        if case["stage"] > 0:
            b.run(max_rounds=40)
            for r in handles:
                r.set_state("lnf", np.full(r.h, 2.0 ** -case["stage"]))
                r.set_state("H", _zeros_like_state(r, "H"))
        b.run(max_rounds=2)
        return dict(case=case, b=b, handles=handles)
    if kind == "whole":
        r = R.REWL(case["model"], case["L"], case["windows"], OVERLAP, case["walkers"],
                   case["lnf_final"], 0.8, seed=_seed(seed))
        return dict(case=case, r=r)
    if kind == "join":
        return dict(case=case, r=_finished(case, seed))
    if kind == "em":
        r = _finished(case, seed, interval=1000)
        r.set_param("production", 1)
        r.set_param("measure_em", 1)
        r.run(max_rounds=200)
        return dict(case=case, r=r)
    if kind == "thermo":
        lng, T = (torch.from_numpy(a).cuda() for a in _thermo_inputs(case, seed))
        return dict(case=case, lng=lng, T=T, U=torch.zeros_like(T), C=torch.zeros_like(T))
    P, X, T = (torch.from_numpy(a).cuda() for a in _train_inputs(case, seed))
    work = torch.zeros(R.mlp_workspace_floats(X.shape[0]), dtype=torch.float32, device="cuda")
    return dict(case=case, P=P, X=X, T=T, m=torch.zeros_like(P), v=torch.zeros_like(P),
                grad=torch.zeros_like(P), work=work, loss=torch.zeros(1, device="cuda"), t=0)


# ------------------------------------------------------------------------------- one pass
def _walkers(r, fields=("spins", "k", "lng", "H", "acc", "lnf", "iter")):
    return {f: r.get_state(f) for f in fields}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "rounds":
        state["r"].run(max_rounds=case["rounds"])
        return _walkers(state["r"])
    if kind == "batch":
        state["b"].run(max_rounds=case["rounds"])
        # each instance's window ln g, and where its walkers are
        return {f: np.concatenate([h.get_state(f).ravel() for h in state["handles"]])
                for f in ("lng_mean", "k", "lnf", "acc")}
    if kind == "start":
        state["r"].init()
        return _walkers(state["r"], ("spins", "k", "pstep", "prep_restarts"))
    if kind == "whole":
        r = state["r"]
        r.init()
        r.run(max_rounds=case["max_rounds"])
        lng, joins = r.stitch()
        return dict(lng=lng, joins=joins, **_walkers(r, ("spins", "k", "lng_mean", "lnf", "acc")))
    if kind == "join":
        lng, joins = state["r"].stitch()
        return dict(lng=lng, joins=joins, error=state["r"].jackknife())
    if kind == "em":
        state["r"].run(max_rounds=case["rounds"])
        lng, joins = state["r"].stitch_em()
        return dict(lng=lng, joins=joins, hist=state["r"].hist_em())
    if kind == "thermo":
        R.thermo(state["lng"], case["model"], case["L"], state["T"], state["U"], state["C"])
        return dict(U=state["U"], C=state["C"])
    s = state
    R.mlp_train(s["P"], s["X"], s["T"], case["steps"], 3e-3, s["t"], s["m"], s["v"], s["grad"],
                s["work"], s["loss"])
    s["t"] += case["steps"]
    return {f: s[f] for f in ("P", "m", "v", "grad", "loss")}


# ------------------------------------------------------------------------------- what it takes
def _layout_work(d, attempts_per_walker):
    N, B = d["L"] ** 2, _bins(d["model"], d["L"])
    nw = d["windows"] * d["walkers"]
    width = min(B + 1, 4 * B // (d["windows"] + 3) + 1)
    return dict(bytes=2 * nw * (N + 12 * width), flops=OPS_PER_ATTEMPT * nw * attempts_per_walker)


def work(case):
    kind = case["kind"]
    if kind == "rounds":
        return _layout_work(case, case["rounds"] * case["interval"])
    if kind == "batch":
        w = [_layout_work(d, case["rounds"] * case["interval"]) for d in _batch_descs(case, 0)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "whole":  # about 200 rounds to ln f = 1e-6, fewer for a larger last ln f
        return _layout_work(case, 10_000 * 200 * min(1.0, -math.log10(case["lnf_final"]) / 6))
    if kind == "start":  # written lattices; one to a few proposals per site
        w = _layout_work(case, 2 * case["L"] ** 2)
        return dict(bytes=case["windows"] * case["walkers"] * case["L"] ** 2, flops=w["flops"])
    if kind == "join":  # every walker's ln g twice (as it is, and as kept for the resampling)
        nw, B = case["windows"] * case["walkers"], _bins(case["model"], case["L"])
        width = min(B + 1, 4 * B // (case["windows"] + 3) + 1)
        return dict(bytes=2 * 8 * nw * width + 8 * 2 * (B + 1),
                    flops=20 * (case["walkers"] + 1) * (B + 1))
    if kind == "em":
        d = dict(case, model=0)
        w = _layout_work(d, case["rounds"] * 1000)
        N = case["L"] ** 2
        return dict(bytes=w["bytes"] + 12 * (N + 1) * (N + 1), flops=w["flops"])
    if kind == "thermo":
        B = _bins(case["model"], case["L"])
        return dict(bytes=8 * (B + 1) + 24 * case["temperatures"],
                    flops=40 * (B + 1) * case["temperatures"])
    n, steps = case["samples"], case["steps"]
    return dict(bytes=steps * (16 * n + 5 * 4 * R.MLP_NPARAM), flops=steps * n * 6 * 4400)


# ------------------------------------------------------------------------------- 64 bits
def _exact_thermo(case, seed):
    lng, T = _thermo_inputs(case, seed)
    model, N = case["model"], case["L"] ** 2
    E = -2.0 * N + (4.0 if model == 0 else 1.0) * np.arange(lng.size)
    U, C = np.zeros(T.size), np.zeros(T.size)
    for i, t in enumerate(T):
        x = lng - E / t
        w = np.exp(x - x.max())
        w /= w.sum()
        u = (w * E).sum()
        U[i], C[i] = u / N, (w * (E - u) ** 2).sum() / (N * t * t)
    return dict(U=U, C=C)


def _exact_train(case, seed):
    P, X, T = (torch.from_numpy(a).double() for a in _train_inputs(case, seed))
    if torch.cuda.is_available():
        P, X, T = P.cuda(), X.cuda(), T.cuda()
    m, v = torch.zeros_like(P), torch.zeros_like(P)
    n = X.shape[0]
    for t in range(1, case["steps"] + 1):
        W1, b1, W2 = P[:192].view(64, 3), P[192:256], P[256:4352].view(64, 64)
        b2, W3, b3 = P[4352:4416], P[4416:4480], P[4480]
        h1 = torch.tanh(X @ W1.T + b1)
        h2 = torch.tanh(h1 @ W2.T + b2)
        r = h2 @ W3 + b3 - T
        loss = (r * r).mean()
        dy = 2.0 * r / n
        dz2 = dy[:, None] * W3 * (1 - h2 * h2)
        dz1 = (dz2 @ W2) * (1 - h1 * h1)
        g = torch.cat([(dz1.T @ X).reshape(-1), dz1.sum(0), (dz2.T @ h1).reshape(-1), dz2.sum(0),
                       h2.T @ dy, dy.sum().reshape(1)])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        P = P - 3e-3 * (m / (1 - 0.9 ** t)) / (torch.sqrt(v / (1 - 0.999 ** t)) + 1e-8)
    return dict(P=P, m=m, v=v, grad=g, loss=loss.reshape(1))


def exact(case, seed):
    if case["kind"] == "thermo":
        return _exact_thermo(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    return None  # a walk's float64 state is defined by its order of operations alone
