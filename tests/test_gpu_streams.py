"""Calls on streams of their own, beside a busy default stream."""
import numpy as np
import pytest
import torch

import paper_2603_01122_gb300 as pm

pytestmark = pytest.mark.gpu


def test_batch_made_behind_a_busy_default_stream():
    """The batch's counters are zeroed on the default stream; a prediction on a
    stream of its own, which does not wait for that one, finds them at zero."""
    torch.cuda.synchronize()
    rng = np.random.default_rng(2)
    n, N, T, W = 3, 2000, 12, 40
    goals = [torch.tensor(rng.uniform(-3, 3, (2, 2)).astype(np.float32)).cuda() for _ in range(n)]
    beta = torch.tensor([0.5, 2.0]).cuda()
    belief = torch.full((4,), float(-np.log(4.0))).cuda()
    z0 = torch.zeros((n, 2), device="cuda")
    counts = torch.full((n, T, W, W), 7, dtype=torch.int32, device="cuda")
    oob = torch.full((n, T), 7, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    ctx = pm.pm_create(0)
    try:
        model = pm.make_model(8, 1.0, 0.1, goals[0], beta)
        torch.cuda.synchronize()
        torch.cuda._sleep(200_000_000)  # the default stream stays busy for about 0.1 s
        batch = pm.pm_batch_create(ctx, model, n)
        grid = pm.make_grid(-2.0, -2.0, 0.1, W, W)
        pm.pm_batch_set(batch, [pm.make_human(goals[i], beta, belief, z0[i], N, T, grid, 7, i, counts[i], oob[i])
                                for i in range(n)], side)
        pm.pm_batch_predict(batch, side)
        side.synchronize()
        total = counts.sum((2, 3)) + oob
        torch.cuda.synchronize()
        assert bool((total == N).all())
        pm.pm_batch_destroy(batch)
    finally:
        pm.pm_destroy(ctx)
