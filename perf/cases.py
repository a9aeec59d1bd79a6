"""What a user of this framework has it do, as measurable cases.

A case is a dict of plain sizes and options; ``prepare`` builds what a program
holds before the call (device tensors, a context, a batch, a captured frame),
``run`` makes one pass through the public entry points and returns every
output, ``work`` says what a pass cannot do without, and ``exact`` gives the
floating-point outputs in 64 bits from plain numpy / torch.

Kinds
  predict  belief update over the observed steps, then the occupancy
           prediction of one human, device buffers in and out
  host     the same from host buffers (what a robot-side caller holds)
  belief   the belief update alone
  batch    many humans: update and prediction of all of them
  frame    a serving frame: newest step of every live human copied in, update,
           prediction in a window around each human, blur and union on the
           room grid, all in one captured graph
  fit      marginal log-likelihood of observed trajectories and its gradient
  planner  blur of one human's occupancy, then the MPPI solve against it

Histories are walks drawn from the model itself (Eq. 2), so beliefs and
rollouts meet the values they meet in use.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2603_01122_gb300 as pm
from paper_2603_01122_gb300.autograd import marginal_loglik

TAU = 2.0 * math.pi


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def _predict(name, **kw):
    case = dict(name=name, kind="predict", K=36, speeds="", heading_off=0, speed_off=0, G=3, B=10, b_lo=-2.0,
                b_hi=2.0, dt=0.02, room=10.0, n_obs=50, N=100_000, T=150, W=200, H=200, res=0.05)
    case.update(kw)
    return case


def listed():
    """Twelve cases, smallest to largest kinds of use."""
    return [
        # the smallest prediction in use: a coarse model of one human, where a
        # call's latency and launches are what a 100 Hz loop pays
        _predict("small", K=8, G=2, B=3, b_lo=-1.0, b_hi=1.0, dt=0.1, room=6.0, n_obs=20, N=10_000, T=20,
                 W=100, H=100, res=0.1),
        # the paper's running example (Table 1): 96 controls, 8192 particles
        _predict("table", K=32, speeds="0.5,1,1.5", G=10, B=5, b_lo=-1.0, b_hi=1.0, dt=0.1, room=5.0, n_obs=20,
                 N=8192, T=10, W=50, H=50, res=0.1),
        # one human at full scale: 100k particles over 3 s, 5 cm cells
        _predict("person"),
        # a model with a heading count of its own and some headings disabled,
        # odd sizes everywhere, goals close enough to be reached
        _predict("masked", K=20, heading_off=0b1001_0000_0000_0001_1000, G=4, B=7, b_lo=-1.0, b_hi=2.0, dt=0.04,
                 room=4.0, n_obs=33, N=30_011, T=75, W=91, H=73, res=0.07),
        # one human with walking speeds to choose from (|U| = 96) at full scale
        _predict("speeds", K=32, speeds="0.5,1,1.5"),
        # the same prediction called from host buffers, results read back
        dict(name="hosted", kind="host", K=36, speeds="", heading_off=0, speed_off=0, G=4, B=10, b_lo=-2.0, b_hi=2.0,
             dt=0.02, room=10.0, n_obs=50, N=50_000, T=100, W=200, H=200, res=0.05),
        # a long history over the largest belief table, at start-up or re-admission
        dict(name="history", kind="belief", K=64, speeds="", heading_off=0, speed_off=0, G=16, B=16, b_lo=-2.0,
             b_hi=2.0, dt=0.05, room=12.0, n_obs=200),
        # a crowd of coarse humans in one batch
        dict(name="crowd", kind="batch", layout=11, n=64, K=8, speeds="", G_lo=2, G_hi=2, B=3, b_lo=-1.0, b_hi=1.0,
             dt=0.1, room=6.0, n_obs=20, N_lo=10_000, N_hi=10_000, T_lo=20, T_hi=20, W=100, H=100, res=0.1),
        # sixteen different humans on a shared room grid
        dict(name="room", kind="batch", layout=20, n=16, K=36, speeds="", G_lo=2, G_hi=6, B=10, b_lo=-2.0, b_hi=2.0,
             dt=0.02, room=20.0, n_obs=50, N_lo=20_000, N_hi=200_000, T_lo=50, T_hi=300, W=400, H=400, res=0.05),
        # a serving frame of 64 live humans, with the planner's union grid
        dict(name="frame", kind="frame", layout=30, n=64, K=36, speeds="", G_lo=2, G_hi=6, B=10, b_lo=-2.0, b_hi=2.0,
             dt=0.02, room=20.0, N=50_000, T=150, window=121, W=400, H=400, res=0.05, sigma=1.5),
        # fitting goals, speed and weights to 256 recorded trajectories
        dict(name="fit", kind="fit", layout=40, M=256, len_lo=50, len_hi=200, K=36, speeds="", G=4, B=10, b_lo=-1.0,
             b_hi=1.0, dt=0.05, room=10.0),
        # the local planner's step: smoothed occupancy, then 8192 sampled controls
        dict(name="planner", kind="planner", T=150, W=200, H=200, res=0.05, N=50_000, sigma=1.5, samples=8192,
             steps=30, stride=5),
    ]


def _log(rng, lo, hi):
    """A whole number, uniform in its logarithm over [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["predict"] * 5 + ["batch"] * 3 + ["frame", "fit", "belief", "host", "planner"])
    speeds = rng.choice(["", "", "0.5,1", "0.5,1,1.5"])
    K = rng.choice([16, 32, 36]) if speeds else rng.choice([8, 16, 20, 24, 36, 36, 64])
    W, H, res = rng.randint(41, 240), rng.randint(41, 240), rng.choice([0.05, 0.1])
    model = dict(K=K, speeds=speeds, b_lo=rng.choice([-2.0, -1.0]), b_hi=rng.choice([1.0, 2.0]),
                 dt=rng.choice([0.02, 0.04, 0.1]), room=rng.choice([6.0, 10.0, 20.0]))
    if kind in ("predict", "host"):
        off = rng.getrandbits(K) & rng.getrandbits(K) & rng.getrandbits(K) if not speeds and rng.random() < 0.3 else 0
        soff = 6 & ((1 << len(speeds.split(","))) - 1) if speeds and rng.random() < 0.3 else 0
        return dict(model, kind=kind, heading_off=off, speed_off=soff, G=rng.randint(1, 10), B=rng.randint(1, 10),
                    n_obs=_log(rng, 1, 200), N=_log(rng, 1000, 100_000), T=_log(rng, 5, 200), W=W, H=H, res=res)
    if kind == "belief":
        G = rng.randint(1, 16)
        return dict(model, kind=kind, heading_off=0, speed_off=0, G=G, B=rng.randint(1, 16), n_obs=_log(rng, 1, 400))
    if kind == "batch":
        n = _log(rng, 2, 64)
        hi = 2_000_000 // n  # all humans together: at most 2M particles over 100 steps
        return dict(model, kind=kind, layout=rng.randint(0, 1 << 20), n=n, G_lo=1, G_hi=6, B=rng.randint(2, 10),
                    n_obs=_log(rng, 1, 60), N_lo=1000, N_hi=min(hi, 150_000), T_lo=5, T_hi=100, W=W, H=H, res=res)
    if kind == "frame":
        return dict(model, kind=kind, speeds="", K=rng.choice([16, 36]), layout=rng.randint(0, 1 << 20),
                    n=rng.randint(1, 40), G_lo=2, G_hi=6, B=10, N=_log(rng, 5000, 50_000), T=rng.randint(30, 150),
                    window=2 * rng.randint(30, 60) + 1, W=rng.randint(200, 400), H=rng.randint(200, 400), res=0.05,
                    sigma=rng.choice([0.0, 1.0, 1.5, 2.5]))
    if kind == "fit":
        return dict(model, kind=kind, layout=rng.randint(0, 1 << 20), M=_log(rng, 4, 300), len_lo=20, len_hi=200,
                    G=rng.randint(1, 8), B=rng.randint(1, 10))
    return dict(kind="planner", T=rng.randint(20, 150), W=W, H=H, res=res, N=_log(rng, 1000, 100_000),
                sigma=rng.choice([1.0, 1.5, 3.0]), samples=_log(rng, 500, 20_000), steps=rng.randint(10, 40),
                stride=rng.randint(1, 5))


# ---------------------------------------------------------------------------
# inputs (numpy, from the seed alone)
# ---------------------------------------------------------------------------
def _mults(case):
    return [float(np.float32(m)) for m in case["speeds"].split(",")] if case["speeds"] else [1.0]


def _betas(case):
    return (np.float32(10.0) ** np.linspace(case["b_lo"], case["b_hi"], case["B"])).astype(np.float32)


def _headings(K):
    th = TAU * np.arange(K) / K
    return np.stack([np.cos(th), np.sin(th)], -1)


def _walk(rng, case, goal, beta, start, n):
    """n steps of Eq. 2 for each row of goal [M, 2], beta [M], start [M, 2]: [M, n + 1, 2] float32."""
    s = float(np.float32(case["dt"]))
    on_k = np.array([not (case.get("heading_off", 0) >> k) & 1 for k in range(case["K"])])
    moves = np.concatenate([s * m * _headings(case["K"]) for m in _mults(case)])
    on = np.tile(on_k, len(_mults(case)))
    if case.get("speed_off", 0):
        on &= np.repeat([not (case["speed_off"] >> q) & 1 for q in range(len(_mults(case)))], case["K"])
    moves = moves[on]
    cost = np.hypot(moves[:, 0], moves[:, 1])
    z = np.array(start, np.float64)
    out = np.empty((z.shape[0], n + 1, 2), np.float32)
    out[:, 0] = z
    for t in range(n):
        nxt = z[:, None, :] + moves[None]
        dist = np.hypot(nxt[..., 0] - goal[:, None, 0], nxt[..., 1] - goal[:, None, 1])
        q = -beta[:, None] * (cost[None] + dist)
        c = np.cumsum(np.exp(q - q.max(1, keepdims=True)), 1)
        k = (c <= rng.random((z.shape[0], 1)) * c[:, -1:]).sum(1).clip(max=len(moves) - 1)
        z = nxt[np.arange(z.shape[0]), k]
        out[:, t + 1] = z
    return out


def _person(case, seed):
    """Goals, betas, history and uniform log-prior of one human."""
    rng = np.random.default_rng([seed, 1])
    room = case["room"]
    goals = rng.uniform(0.0, room, (case["G"], 2)).astype(np.float32)
    beta = _betas(case)
    start = rng.uniform(0.2 * room, 0.8 * room, (1, 2))
    g, b = rng.integers(case["G"]), rng.integers(case["B"])
    obs = _walk(rng, case, goals[g:g + 1].astype(np.float64), beta[b:b + 1].astype(np.float64), start, case["n_obs"])[0]
    J = case["G"] * case["B"]
    return dict(goals=goals, beta=beta, obs=obs, prior=np.full(J, -math.log(J), np.float32), start=start[0])


def _origin(case, at):
    """Origin of a grid centred on the start."""
    return [float(np.float32(at[0] - 0.5 * case["W"] * case["res"])),
            float(np.float32(at[1] - 0.5 * case["H"] * case["res"]))]


def _people(case, seed):
    """The humans of a batch: sizes from the case's layout, values from the seed."""
    lay = np.random.default_rng([case["layout"], 7])
    G = lay.integers(case["G_lo"], case["G_hi"] + 1, case["n"])
    frame = case["kind"] == "frame"
    N = np.full(case["n"], case["N"]) if frame else \
        np.exp(lay.uniform(np.log(case["N_lo"]), np.log(case["N_hi"]), case["n"])).round().astype(int)
    T = np.full(case["n"], case["T"]) if frame else lay.integers(case["T_lo"], case["T_hi"] + 1, case["n"])
    rng = np.random.default_rng([seed, 2])
    room, n = case["room"], case["n"]
    beta = _betas(case)
    goals = [rng.uniform(0.0, room, (g, 2)).astype(np.float32) for g in G]
    to = np.array([gs[rng.integers(len(gs))] for gs in goals], np.float64)
    bt = beta[rng.integers(case["B"], size=n)].astype(np.float64)
    start = rng.uniform(0.2 * room, 0.8 * room, (n, 2))
    steps = 51 if frame else case["n_obs"]
    path = _walk(rng, case, to, bt, start, steps)
    priors = []
    for i in range(n):
        lp = np.full(len(goals[i]) * case["B"], -math.log(len(goals[i]) * case["B"]))
        if frame:  # a live human's belief before its newest step
            lp = _posterior64(case, goals[i], beta, path[i, :steps], lp)
        priors.append(lp.astype(np.float32))
    obs = path[:, steps - 1:] if frame else path
    return dict(G=G, N=N, T=T, goals=goals, beta=beta, obs=obs, priors=priors)


def _tracks(case, seed):
    """Observed trajectories of different lengths, as CSR."""
    lay = np.random.default_rng([case["layout"], 9])
    lengths = lay.integers(case["len_lo"], case["len_hi"] + 1, case["M"])
    rng = np.random.default_rng([seed, 3])
    goals = rng.uniform(0.0, case["room"], (case["G"], 2)).astype(np.float32)
    to = goals[rng.integers(case["G"], size=case["M"])].astype(np.float64)
    bt = 10.0 ** rng.uniform(case["b_lo"], case["b_hi"], case["M"])
    path = _walk(rng, case, to, bt, rng.uniform(0.0, case["room"], (case["M"], 2)), case["len_hi"])
    # recorded positions carry a little sensor noise
    path += rng.normal(0.0, 0.05 * case["dt"], path.shape).astype(np.float32)
    traj = np.concatenate([path[i, :n + 1] for i, n in enumerate(lengths)])
    off = np.concatenate([[0], np.cumsum(lengths + 1)]).astype(np.int32)
    J = case["G"] * case["B"]
    return dict(goals=goals, beta=_betas(case), traj=traj, offsets=off, lengths=lengths,
                prior=np.full(J, -math.log(J), np.float32))


def _plan(case, seed):
    """Counts of a spreading cloud of N particles, and a planner's samples."""
    rng = np.random.default_rng([seed, 4])
    T, H, W, n = case["T"], case["H"], case["W"], min(case["N"], 4000)
    at = rng.uniform(0.3, 0.7, 2) * (W, H) * case["res"]
    step = rng.normal(0.0, 0.02, (T, n, 2)) + rng.uniform(-0.012, 0.012, (1, n, 2))
    cell = np.floor((at + np.cumsum(step, 0)) / case["res"]).astype(np.int64)
    ok = (cell[..., 0] >= 0) & (cell[..., 0] < W) & (cell[..., 1] >= 0) & (cell[..., 1] < H)
    flat = (np.arange(T)[:, None] * H + cell[..., 1]) * W + cell[..., 0]
    counts = np.bincount(flat[ok], minlength=T * H * W).reshape(T, H, W)
    counts = (counts * (case["N"] // n)).astype(np.int32)
    z0 = [float(np.float32(v)) for v in (*(rng.uniform(0.1, 0.9, 2) * (W, H) * case["res"]), 0.8,
                                         rng.uniform(-3.0, 3.0))]
    u_ref = rng.normal(0.0, 0.1, (case["steps"], 2)).astype(np.float32)
    delta = rng.normal(0.0, 0.4, (case["steps"], case["samples"], 2)).astype(np.float32)
    goal = [float(np.float32(v)) for v in (*(rng.uniform(0.1, 0.9, 2) * (W, H) * case["res"]), 0.0, 0.0)]
    return dict(counts=counts, z0=z0, u_ref=u_ref, delta=delta, goal=goal)


MPPI = dict(dt=0.1, q=(1.0, 1.0, 0.1, 0.0), q_final=(10.0, 10.0, 0.5, 0.0), r=(0.05, 0.02), coll_threshold=0.002,
            coll_cost=20.0, step_cost=0.1, temperature=5.0)


# ---------------------------------------------------------------------------
# what a program holds before the call
# ---------------------------------------------------------------------------
class _Held:
    """Tensors, a context and a batch, released together."""

    def __init__(self, case):
        self.case = case
        self.ctx = pm.pm_create(0)
        self.batch = None
        self.graph = None

    def __del__(self):
        try:
            torch.cuda.synchronize()
            self.graph = None
            if self.batch is not None:
                pm.pm_batch_destroy(self.batch)
            pm.pm_destroy(self.ctx)
        except Exception:  # the interpreter or the driver is going away
            pass


def _dev(a):
    return torch.as_tensor(a).cuda()


def _model(case, goals, beta):
    return pm.make_model(case["K"], 1.0, case["dt"], goals, beta, heading_off=case.get("heading_off", 0),
                         speeds=_mults(case) if case["speeds"] else None, speed_off=case.get("speed_off", 0))


def prepare(case, seed):
    st = _Held(case)
    kind = case["kind"]
    st.seed = int(seed) & 0x7FFFFFFF
    if kind in ("predict", "belief", "host"):
        p = _person(case, seed)
        st.n_obs = case["n_obs"]
        if kind == "host":
            pin = {k: torch.as_tensor(p[k]).pin_memory() for k in ("goals", "beta", "obs", "prior")}
            st.goals, st.beta, st.obs, st.prior = pin["goals"], pin["beta"], pin["obs"], pin["prior"]
            st.post = torch.empty_like(st.prior).pin_memory()
            st.counts = torch.empty((case["T"], case["H"], case["W"]), dtype=torch.int32).pin_memory()
            st.oob = torch.empty(case["T"], dtype=torch.int32).pin_memory()
        else:
            st.goals, st.beta, st.obs, st.prior = (_dev(p[k]) for k in ("goals", "beta", "obs", "prior"))
            st.post = torch.empty_like(st.prior)
            if kind == "predict":
                st.counts = torch.empty((case["T"], case["H"], case["W"]), dtype=torch.int32, device="cuda")
                st.oob = torch.empty(case["T"], dtype=torch.int32, device="cuda")
        st.model = _model(case, st.goals, st.beta)
        if kind != "belief":
            st.z0 = [float(v) for v in p["obs"][-1]]
            st.grid = pm.make_grid(*_origin(case, p["start"]), case["res"], case["W"], case["H"])
    elif kind in ("batch", "frame"):
        _prepare_batch(st, case, seed)
    elif kind == "fit":
        p = _tracks(case, seed)
        st.goals = _dev(p["goals"]).requires_grad_()
        st.speed = torch.tensor(1.0, device="cuda").requires_grad_()
        st.w = torch.tensor([1.0, 1.0], device="cuda").requires_grad_()
        st.beta, st.off, st.traj, st.prior = (_dev(p[k]) for k in ("beta", "offsets", "traj", "prior"))
        st.mults = _mults(case) if case["speeds"] else None
    else:
        p = _plan(case, seed)
        st.counts, st.u_ref, st.delta = (_dev(p[k]) for k in ("counts", "u_ref", "delta"))
        st.z0 = p["z0"]
        st.grid = pm.make_grid(0.0, 0.0, case["res"], case["W"], case["H"])
        st.prob = torch.empty((case["T"], case["H"], case["W"]), device="cuda")
        st.params = pm.make_mppi(case["samples"], case["steps"], pred_stride=case["stride"], goal=p["goal"], **MPPI)
        st.ctg = torch.empty((case["steps"], case["samples"]), device="cuda")
        st.u_opt = torch.empty((case["steps"], 2), device="cuda")
    torch.cuda.synchronize()
    return st


def _prepare_batch(st, case, seed):
    p = _people(case, seed)
    frame, n = case["kind"] == "frame", case["n"]
    st.sizes = [len(lp) for lp in p["priors"]]
    st.prior = _dev(np.concatenate(p["priors"]))
    st.post = torch.empty_like(st.prior)
    st.beta = _dev(p["beta"])
    st.goals = [_dev(g) for g in p["goals"]]
    st.obs_host = torch.as_tensor(np.ascontiguousarray(p["obs"])).pin_memory()
    st.obs = st.obs_host.cuda()
    side = (case["window"], case["window"]) if frame else (case["H"], case["W"])
    T = [int(t) for t in p["T"]]  # the humans' histograms one after another, [T_i][H][W] each
    st.counts = torch.empty((sum(T), *side), dtype=torch.int32, device="cuda")
    st.oob = torch.empty(sum(T), dtype=torch.int32, device="cuda")
    counts, oob = st.counts.split(T), st.oob.split(T)
    shared = pm.make_model(case["K"], 1.0, case["dt"], st.goals[0], st.beta,
                           speeds=_mults(case) if case["speeds"] else None)
    st.batch = pm.pm_batch_create(st.ctx, shared, n)
    stream = torch.cuda.current_stream()
    if frame:
        pm.pm_batch_set_zeroing(st.batch, 1, stream)
        pm.pm_batch_set_block_flags(st.batch, 1, stream)
    grid = pm.make_grid(0.0, 0.0, case["res"], side[1], side[0])
    beliefs = st.post.split(st.sizes)
    humans = [pm.make_human(st.goals[i], st.beta, beliefs[i], st.obs[i, -1], int(p["N"][i]), T[i], grid, st.seed,
                            100 + i, counts[i], oob[i], obs_xy=st.obs[i],
                            n_obs=st.obs.shape[1] - 1, center=int(frame)) for i in range(n)]
    pm.pm_batch_set(st.batch, humans, stream)
    if not frame:
        return
    st.union_grid = pm.make_grid(0.0, 0.0, case["res"], case["W"], case["H"])
    st.union = torch.empty((case["T"], case["H"], case["W"]), device="cuda")
    torch.cuda.synchronize()
    main, aside = torch.cuda.Stream(), torch.cuda.Stream()
    _frame(st, main, aside)  # before the capture, as a server warms its frame up
    torch.cuda.synchronize()
    st.graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(st.graph, stream=main):
        _frame(st, main, aside)


def _frame(st, main, aside):
    """One serving frame on ``main``, the zeroing beside the belief update on ``aside``."""
    case = st.case
    with torch.cuda.stream(main):
        st.obs.copy_(st.obs_host, non_blocking=True)
        aside.wait_stream(main)
        st.post.copy_(st.prior)
    pm.pm_batch_zero(st.batch, aside)
    pm.pm_batch_update_posterior(st.batch, main)
    main.wait_stream(aside)
    pm.pm_batch_rollout(st.batch, main)
    pm.pm_batch_union(st.batch, case["sigma"], case["T"], st.union_grid, st.union, main)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    case, kind = st.case, st.case["kind"]
    stream = torch.cuda.current_stream()
    if kind in ("predict", "belief"):
        pm.pm_update_posterior_into(st.ctx, st.model, st.obs, st.n_obs, st.prior, st.post, stream)
        if kind == "belief":
            return [st.post]
        pm.pm_predict_occupancy(st.ctx, st.model, st.post, *st.z0, case["N"], case["T"], st.grid, st.seed, 5,
                                st.counts, st.oob, stream)
        return [st.post, st.counts, st.oob]
    if kind == "host":
        pm.pm_predict_host(st.ctx, st.model, st.goals, st.beta, st.obs, st.n_obs, st.prior, case["N"], case["T"],
                           st.grid, st.seed, 5, st.post, st.counts, st.oob, stream)
        return [st.post, st.counts, st.oob]
    if kind == "batch":
        st.post.copy_(st.prior)
        pm.pm_batch_update_posterior(st.batch, stream)
        pm.pm_batch_predict(st.batch, stream)
        return [st.post, st.counts, st.oob]
    if kind == "frame":
        st.graph.replay()
        return [st.post, st.counts, st.oob, st.union]
    if kind == "fit":
        L = marginal_loglik(st.goals, st.speed, st.w, st.beta, case["K"], case["dt"], st.off, st.traj, st.prior,
                            st.ctx, speeds=st.mults)
        grads = torch.autograd.grad(L, (st.goals, st.speed, st.w))
        return [L.detach(), *grads]
    pm.pm_smooth_occupancy(st.ctx, st.counts, case["N"], case["T"], st.grid, case["sigma"], st.prob, stream)
    pm.pm_mppi_solve(st.ctx, st.params, st.z0, st.u_ref, st.delta, st.prob, case["T"], st.grid, st.ctg, st.u_opt,
                     stream)
    return [st.prob, st.ctg, st.u_opt]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _rollout_flops(steps):
    """A particle-step: its share of the random block, the draw, the Euler step and the binning."""
    return 64 * steps


def work(case):
    """Bytes: inputs read once, outputs written once. Flops: ten per control whose value is needed
    (belief and gradient), and a fixed cost per particle-step of a rollout, however many controls
    its draw chooses from."""
    kind = case["kind"]
    U = case["K"] * len(_mults(case)) if "K" in case else 0
    if kind in ("predict", "host", "belief"):
        J = case["G"] * case["B"]
        b = 8 * (case["n_obs"] + 1) + 4 * (2 * case["G"] + case["B"]) + 8 * J
        f = 10 * case["n_obs"] * J * U
        if kind != "belief":
            b += 4 * case["T"] * (case["H"] * case["W"] + 1)
            f += _rollout_flops(case["N"] * case["T"])
        return {"bytes": b, "flops": f}
    if kind in ("batch", "frame"):
        lay = np.random.default_rng([case["layout"], 7])
        G = lay.integers(case["G_lo"], case["G_hi"] + 1, case["n"])
        if kind == "frame":
            N, T, n_obs = np.full(case["n"], case["N"]), np.full(case["n"], case["T"]), 1
            cells, extra = case["window"] ** 2, 4 * case["T"] * case["H"] * case["W"]
        else:
            N = np.exp(lay.uniform(np.log(case["N_lo"]), np.log(case["N_hi"]), case["n"])).round().astype(int)
            T, n_obs = lay.integers(case["T_lo"], case["T_hi"] + 1, case["n"]), case["n_obs"]
            cells, extra = case["W"] * case["H"], 0
        J = int(G.sum()) * case["B"]
        b = case["n"] * 8 * (n_obs + 1) + 8 * int(G.sum()) + 8 * J + 4 * int(T.sum()) * (cells + 1) + extra
        return {"bytes": b, "flops": 10 * n_obs * J * U + _rollout_flops(int((N * T).sum()))}
    if kind == "fit":
        lay = np.random.default_rng([case["layout"], 9])
        steps = int(lay.integers(case["len_lo"], case["len_hi"] + 1, case["M"]).sum())
        return {"bytes": 8 * (steps + case["M"]) + 4 * case["M"], "flops": 20 * steps * U * case["G"] * case["B"]}
    cells = case["T"] * case["H"] * case["W"]
    R = math.ceil(3 * case["sigma"])
    sim = case["samples"] * case["steps"]
    return {"bytes": 8 * cells + 12 * sim, "flops": 4 * (2 * R + 1) * cells + 60 * sim}


# ---------------------------------------------------------------------------
# 64-bit values of the floating-point outputs
# ---------------------------------------------------------------------------
def _posterior64(case, goals, beta, obs, log_prior):
    """Eq. 7 over the steps of obs [n + 1, 2] for every component g * B + b."""
    goals, beta, obs = goals.astype(np.float64), beta.astype(np.float64), obs.astype(np.float64)
    s, mults = float(np.float32(case["dt"])), _mults(case)
    mult_on = [q for q in range(len(mults)) if not (case.get("speed_off", 0) >> q) & 1]
    on_k = np.array([not (case.get("heading_off", 0) >> k) & 1 for k in range(case["K"])])
    moves = np.concatenate([s * mults[q] * _headings(case["K"])[on_k] for q in mult_on])
    cost = np.concatenate([np.full(on_k.sum(), s * mults[q]) for q in mult_on])
    z, d = obs[:-1], np.diff(obs, axis=0)
    step = np.hypot(d[:, 0], d[:, 1])
    z, d, step = z[step >= 1e-6], d[step >= 1e-6], step[step >= 1e-6]
    near = np.abs(np.array([mults[q] for q in mult_on])[None] - step[:, None] / s).argmin(1)
    so = s * np.array([mults[q] for q in mult_on])[near]
    nxt = z[:, None] + moves[None]  # [n, U, 2]
    own = z + d / step[:, None] * so[:, None]
    out = np.array(log_prior, np.float64)
    for g in range(len(goals)):
        Q = -(cost[None] + np.hypot(nxt[..., 0] - goals[g, 0], nxt[..., 1] - goals[g, 1]))
        Qo = -(so + np.hypot(own[:, 0] - goals[g, 0], own[:, 1] - goals[g, 1]))
        for b in range(len(beta)):
            a = beta[b] * (Q - Qo[:, None])
            m = a.max(1, initial=-np.inf) if len(a) else np.zeros(0)
            out[g * len(beta) + b] -= (m + np.log(np.exp(a - m[:, None]).sum(1))).sum()
    m = out.max()
    return out - (m + math.log(np.exp(out - m).sum()))


def _fit64(case, seed):
    p = _tracks(case, seed)
    f64 = dict(dtype=torch.float64)
    goals = torch.tensor(p["goals"], **f64).requires_grad_()
    v = torch.tensor(1.0, **f64).requires_grad_()
    w = torch.tensor([1.0, 1.0], **f64).requires_grad_()
    beta, prior = torch.tensor(p["beta"], **f64), torch.tensor(p["prior"], **f64)
    e_k = torch.tensor(_headings(case["K"]))
    mult = torch.tensor(_mults(case), **f64)
    dt = float(np.float32(case["dt"]))
    total, grads = 0.0, [torch.zeros_like(goals), torch.zeros_like(v), torch.zeros_like(w)]
    U = case["K"] * len(mult)
    for i in range(case["M"]):
        o = torch.tensor(p["traj"][p["offsets"][i]:p["offsets"][i + 1]], **f64)
        z, d = o[:-1], o.diff(dim=0)
        step = d.norm(dim=1)
        keep = step >= 1e-6
        z, d, step = z[keep], d[keep], step[keep]
        m_o = mult[(mult[None] - (step / dt)[:, None]).abs().argmin(1)]
        move = (mult[:, None, None] * e_k[None]).reshape(U, 2) * (v * dt)
        cost = w[0] * (mult[:, None].expand(-1, case["K"]).reshape(U) * (v * dt))
        nxt = (z[:, None] + move[None])[:, None] - goals[None, :, None]  # [n, G, U, 2]
        own = (z + d / step[:, None] * (m_o * v * dt)[:, None])[:, None] - goals[None]
        Q = -(cost + w[1] * torch.linalg.vector_norm(nxt, dim=-1))
        Qo = -((w[0] * m_o * v * dt)[:, None] + w[1] * torch.linalg.vector_norm(own, dim=-1))
        lp = beta[None, None] * Qo[..., None] - torch.logsumexp(beta[None, None, :, None] * Q[:, :, None], -1)
        L = torch.logsumexp(lp.sum(0).reshape(-1) + prior, 0)
        for acc, g in zip(grads, torch.autograd.grad(L, (goals, v, w))):
            acc += g
        total += float(L.detach())
    return [torch.tensor(total, **f64), *grads]


def _planner64(case, seed):
    p = _plan(case, seed)
    sigma, R = float(np.float32(case["sigma"])), math.ceil(3 * float(np.float32(case["sigma"])))
    i = np.arange(-R, R + 1)
    taps = np.exp(-i * i / (2 * sigma * sigma)) if R else np.ones(1)
    taps /= taps.sum()
    prob = torch.tensor(p["counts"], dtype=torch.float64) / case["N"]
    for axis, (a, b) in ((2, (0, R)), (1, (R, 0))):
        pad = torch.nn.functional.pad(prob, (b, b, a, a))
        n = prob.shape[axis]
        prob = sum(float(taps[k]) * pad.narrow(axis, k, n) for k in range(2 * R + 1))
    prob = prob.numpy()
    T, N, f = case["steps"], case["samples"], np.float32
    u = p["u_ref"].astype(np.float64)[:, None] + p["delta"].astype(np.float64)
    x, y, v, th = (np.full(N, c) for c in p["z0"])
    q, qf, r = (np.array([float(f(c)) for c in MPPI[k]]) for k in ("q", "q_final", "r"))
    dt, goal, res = float(f(MPPI["dt"])), np.array(p["goal"]), float(f(case["res"]))
    run = np.empty((T, N))
    for t in range(T):
        x, y, v, th = x + v * np.cos(th) * dt, y + v * np.sin(th) * dt, v + u[t, :, 0] * dt, th + u[t, :, 1] * dt
        e = np.stack([x, y, v, th]) - goal[:, None]
        run[t] = (q[:, None] * e * e).sum(0) + (r[None] * u[t] ** 2).sum(1) + float(f(MPPI["step_cost"]))
        k = (t + 1) * case["stride"] - 1
        if k < case["T"]:
            cx, cy = np.floor(x / res).astype(int), np.floor(y / res).astype(int)
            ok = (cx >= 0) & (cx < case["W"]) & (cy >= 0) & (cy < case["H"])
            hit = prob[k, cy.clip(0, case["H"] - 1), cx.clip(0, case["W"] - 1)] >= float(f(MPPI["coll_threshold"]))
            run[t] += np.where(ok & hit, MPPI["coll_cost"], 0.0)
    e = np.stack([x, y, v, th]) - goal[:, None]
    ctg = np.cumsum(run[::-1], 0)[::-1] + (qf[:, None] * e * e).sum(0)
    wgt = np.exp(-(ctg - ctg.min(1, keepdims=True)) / MPPI["temperature"])
    d64 = p["delta"].astype(np.float64)
    u_opt = p["u_ref"].astype(np.float64) + (wgt[..., None] * d64).sum(1) / wgt.sum(1)[:, None]
    return [torch.tensor(prob), torch.tensor(ctg.copy()), torch.tensor(u_opt)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("predict", "host", "belief"):
        p = _person(case, seed)
        post = torch.tensor(_posterior64(case, p["goals"], p["beta"], p["obs"], p["prior"]))
        return [post] if kind == "belief" else [post, None, None]
    if kind in ("batch", "frame"):
        p = _people(case, seed)
        post = torch.tensor(np.concatenate([_posterior64(case, p["goals"][i], p["beta"], p["obs"][i], p["priors"][i])
                                            for i in range(case["n"])]))
        return [post, None, None] if kind == "batch" else [post, None, None, None]
    return _fit64(case, seed) if kind == "fit" else _planner64(case, seed)
