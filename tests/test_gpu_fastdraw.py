"""The closed-form heading draw against the weight-by-weight draw.

A model with more than 16 beta values takes the weight-by-weight draw at every
step. Padding a smaller model's beta grid to 17 values whose added components
have a log-belief of -inf leaves every random choice as it is, so the two calls
must agree in every count: no tolerance.
"""
import numpy as np
import pytest
import torch

import paper_2603_01122_gb300 as pm

pytestmark = pytest.mark.gpu


def _predict(K, speeds, speed_off, goals, beta, log_b, dt, N, T, W, H, res, z0, traced):
    ctx = pm.pm_create(0)
    try:
        g, b = torch.tensor(goals).cuda(), torch.tensor(beta).cuda()
        model = pm.make_model(K, 1.0, dt, g, b, speeds=speeds, speed_off=speed_off)
        lb = torch.tensor(log_b).cuda()
        counts = torch.empty((T, H, W), dtype=torch.int32, device="cuda")
        oob = torch.empty(T, dtype=torch.int32, device="cuda")
        grid = pm.make_grid(z0[0] - 0.5 * W * res, z0[1] - 0.5 * H * res, res, W, H)
        if traced:
            states = torch.empty((N, T, 2), device="cuda")
            pm.pm_predict_occupancy_traced(ctx, model, lb, *z0, N, T, grid, 7, 3, counts, oob, N, states, None, None)
        else:
            pm.pm_predict_occupancy(ctx, model, lb, *z0, N, T, grid, 7, 3, counts, oob)
        pm.pm_sync_status(ctx)
        out = [counts.cpu().numpy(), oob.cpu().numpy()]
        return out + [states.cpu().numpy()] if traced else out
    finally:
        pm.pm_destroy(ctx)


@pytest.mark.parametrize("K,speeds,off,dt,b_lo,b_hi,near", [
    (20, None, 0, 0.02, -2.0, 2.0, False),   # the fewest headings
    (23, None, 0, 0.05, -2.0, 1.0, False),   # odd, not a template size
    (36, None, 0, 0.02, -2.0, 2.0, True),    # goals reached: both forms in turn
    (64, None, 0, 0.1, -2.0, 1.0, True),
    (36, None, 0, 0.1, -2.0, 2.0, False),    # some rows beyond the usable kappa
    (16, (0.5, 1.0), 0, 0.04, -1.0, 1.0, False),
    (32, (0.5, 1.0, 1.5), 0, 0.02, -2.0, 2.0, True),
    (20, (0.25, 1.0, 1.5, 2.0), 0b0101, 0.04, -1.0, 1.0, False),
    (36, (0.5, 1.0), 0b10, 0.04, -2.0, 1.0, False),  # one speed left
])
@pytest.mark.parametrize("traced", [False, True])
def test_equals_weight_by_weight(K, speeds, off, dt, b_lo, b_hi, near, traced):
    rng = np.random.default_rng(K)
    G, B, N, T, W, H, res, z0 = 3, 16, 3001, 61, 83, 77, 0.07, (1.5, -0.5)
    goals = (np.array(z0) + rng.uniform(-1.0, 1.0, (G, 2)) * (0.5 if near else 8.0)).astype(np.float32)
    beta = (10.0 ** np.linspace(b_lo, b_hi, B)).astype(np.float32)
    beta[3] = -beta[3]  # a pedestrian walking away from the goal
    beta[5] = 0.0
    log_b = np.log(rng.dirichlet(np.ones(G * B))).astype(np.float32)
    wide = np.full((G, B + 1), -np.inf, np.float32)
    wide[:, :B] = log_b.reshape(G, B)
    args = (dt, N, T, W, H, res, z0, traced)
    got = _predict(K, speeds, off, goals, beta, log_b, *args)
    want = _predict(K, speeds, off, goals, np.append(beta, np.float32(1.0)), wide.ravel(), *args)
    assert got[0].sum() + got[1].sum() == N * T
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("K,speeds,off", [(36, None, 0), (20, None, 0), (64, None, 0), (32, (0.5, 1.0, 1.5), 0),
                                          (16, (0.5, 1.0, 1.5), 0b110)])  # the last: too few controls left for rows
@pytest.mark.parametrize("marks", [0, 1])
def test_batch_equals_weight_by_weight(K, speeds, off, marks):
    rng = np.random.default_rng(K + 1)
    n, B, T, W, H = 5, 9, 40, 61, 67
    outs = []
    goals = [torch.tensor(rng.uniform(-4.0, 4.0, (1 + i % 3, 2)).astype(np.float32)).cuda() for i in range(n)]
    beta = (10.0 ** np.linspace(-2.0, 2.0, B)).astype(np.float32)
    belief = [np.log(rng.dirichlet(np.ones(len(g) * B))).astype(np.float32).reshape(len(g), B) for g in goals]
    for pad in (0, 17 - B):
        ctx = pm.pm_create(0)
        try:
            b = torch.tensor(np.append(beta, np.ones(pad, np.float32))).cuda()
            model = pm.make_model(K, 1.0, 0.03, goals[0], b, speeds=speeds, speed_off=off)
            batch = pm.pm_batch_create(ctx, model, n)
            z0 = torch.zeros((n, 2), device="cuda")
            lb = [torch.tensor(np.pad(p, ((0, 0), (0, pad)), constant_values=-np.inf).ravel()).cuda() for p in belief]
            counts = torch.empty((n, T, H, W), dtype=torch.int32, device="cuda")
            oob = torch.empty((n, T), dtype=torch.int32, device="cuda")
            grid = pm.make_grid(-2.0, -2.0, 0.06, W, H)
            if marks:
                pm.pm_batch_set_block_flags(batch, 1)
            pm.pm_batch_set(batch, [pm.make_human(goals[i], b, lb[i], z0[i], 500 + 333 * i, T, grid, 7, i, counts[i],
                                                  oob[i]) for i in range(n)])
            pm.pm_batch_predict(batch)
            pm.pm_sync_status(ctx)
            outs.append((counts.cpu().numpy(), oob.cpu().numpy()))
            pm.pm_batch_destroy(batch)
        finally:
            pm.pm_destroy(ctx)
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])


@pytest.mark.parametrize("K,speeds", [(20, None), (36, None), (64, None), (32, (0.5, 1.0, 1.5))])
@pytest.mark.parametrize("away", [1e3, 1e4, 3e5, 1e7])
def test_far_goals_equal_weight_by_weight(K, speeds, away):
    """Goals so far away that the rounding of beta |z - g| shows in the fixed-point weights."""
    rng = np.random.default_rng(K)
    G, B, N, T, W, H, res, z0 = 2, 16, 6001, 33, 61, 61, 0.1, (1.5, -0.5)
    goals = (np.array(z0) + away * np.array([[0.6, 0.8], [-1.0, 0.3]])).astype(np.float32)
    beta = (10.0 ** np.linspace(-2.0, 1.5, B)).astype(np.float32)
    beta[::3] *= -1.0
    log_b = np.log(rng.dirichlet(np.ones(G * B))).astype(np.float32)
    wide = np.full((G, B + 1), -np.inf, np.float32)
    wide[:, :B] = log_b.reshape(G, B)
    args = (0.05, N, T, W, H, res, z0, True)
    got = _predict(K, speeds, 0, goals, beta, log_b, *args)
    want = _predict(K, speeds, 0, goals, np.append(beta, np.float32(1.0)), wide.ravel(), *args)
    for a, b in zip(got, want):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("K,speeds,lines", [(36, None, (31, 32, 47, 48)), (20, None, (10, 11, 15, 16, 23, 24)),
                                            (32, (0.5, 1.0, 1.5), (7, 8, 11, 12, 13, 14)),
                                            (36, (0.5, 1.0), (7, 8, 11, 12, 17, 18)),
                                            (12, (0.5, 1.0, 1.5, 2.0), (10, 11, 15, 16, 23, 24))])
@pytest.mark.parametrize("marks", [0, 1])
def test_short_batches_and_captures(K, speeds, lines, marks):
    """Horizons on either side of the lines from which rows are built, in a batch
    and alone; and a graph captured on a short batch, replayed on a longer one."""
    rng = np.random.default_rng(K)
    n, B, N, W, H = 3, 9, 700, 41, 47
    goals = [torch.tensor(rng.uniform(-4.0, 4.0, (2 + i, 2)).astype(np.float32)).cuda() for i in range(n)]
    beta = torch.tensor((10.0 ** np.linspace(-2.0, 1.5, B)).astype(np.float32)).cuda()
    belief = [torch.tensor(np.log(rng.dirichlet(np.ones(len(g) * B))).astype(np.float32)).cuda() for g in goals]
    z0 = torch.zeros((n, 2), device="cuda")
    grid = pm.make_grid(-2.0, -2.0, 0.1, W, H)
    ctx = pm.pm_create(0)
    batch = None
    try:
        model = pm.make_model(K, 1.0, 0.04, goals[0], beta, speeds=speeds)
        batch = pm.pm_batch_create(ctx, model, n)
        if marks:
            pm.pm_batch_set_block_flags(batch, 1)
        graph, stream = None, torch.cuda.Stream()
        for T in lines:
            counts = torch.empty((n, T, H, W), dtype=torch.int32, device="cuda")
            oob = torch.empty((n, T), dtype=torch.int32, device="cuda")
            torch.cuda.synchronize()
            pm.pm_batch_set(batch, [pm.make_human(goals[i], beta, belief[i], z0[i], N, T, grid, 7, i, counts[i], oob[i])
                                    for i in range(n)], stream)
            want = []
            for i in range(n):
                c, o = torch.empty_like(counts[0]), torch.empty_like(oob[0])
                one = pm.make_model(K, 1.0, 0.04, goals[i], beta, speeds=speeds)
                pm.pm_predict_occupancy(ctx, one, belief[i], 0.0, 0.0, N, T, grid, 7, i, c, o, stream)
                want.append((c, o))
            runs = [lambda: pm.pm_batch_predict(batch, stream)]
            stream.synchronize()
            if graph is None:
                pm.pm_batch_predict(batch, stream)
                stream.synchronize()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    pm.pm_batch_predict(batch, stream)
            with torch.cuda.stream(stream):
                runs.append(graph.replay)
                for run in runs:
                    counts.fill_(-1)
                    oob.fill_(-1)
                    run()
                    stream.synchronize()
                    for i, (c, o) in enumerate(want):
                        assert torch.equal(counts[i], c) and torch.equal(oob[i], o), (T, i)
        pm.pm_sync_status(ctx)
    finally:
        if batch is not None:
            pm.pm_batch_destroy(batch)
        pm.pm_destroy(ctx)


@pytest.mark.parametrize("K,speeds", [(20, (0.25, 1.0, 1.5, 2.0)), (36, (0.25, 0.5, 1.0, 1.5)), (32, (0.5, 1.0, 1.5))])
def test_batch_with_own_speed_masks(K, speeds):
    """Each human of a batch disables other speeds; its rows are those of its own
    enabled ones, as in the single-human call with that mask."""
    rng = np.random.default_rng(K)
    S, B, N, T, W, H = len(speeds), 7, 900, 40, 51, 45
    masks = [m for m in range(1 << S) if m != (1 << S) - 1]
    n = len(masks)
    goals = [torch.tensor(rng.uniform(-5.0, 5.0, (2, 2)).astype(np.float32)).cuda() for _ in range(n)]
    beta = torch.tensor((10.0 ** np.linspace(-2.0, 1.5, B)).astype(np.float32)).cuda()
    belief = torch.full((2 * B,), float(-np.log(2 * B))).cuda()
    z0 = torch.zeros((n, 2), device="cuda")
    grid = pm.make_grid(-2.0, -2.0, 0.09, W, H)
    counts = torch.empty((n, T, H, W), dtype=torch.int32, device="cuda")
    oob = torch.empty((n, T), dtype=torch.int32, device="cuda")
    ctx = pm.pm_create(0)
    try:
        batch = pm.pm_batch_create(ctx, pm.make_model(K, 1.0, 0.03, goals[0], beta, speeds=speeds), n)
        pm.pm_batch_set(batch, [pm.make_human(goals[i], beta, belief, z0[i], N, T, grid, 7, i, counts[i], oob[i],
                                              speed_off=masks[i]) for i in range(n)])
        pm.pm_batch_predict(batch)
        for i in range(n):
            c, o = torch.empty_like(counts[0]), torch.empty_like(oob[0])
            one = pm.make_model(K, 1.0, 0.03, goals[i], beta, speeds=speeds, speed_off=masks[i])
            pm.pm_predict_occupancy(ctx, one, belief, 0.0, 0.0, N, T, grid, 7, i, c, o)
            pm.pm_sync_status(ctx)
            assert torch.equal(counts[i], c) and torch.equal(oob[i], o), masks[i]
        pm.pm_batch_destroy(batch)
    finally:
        pm.pm_destroy(ctx)
