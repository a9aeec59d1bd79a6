"""The belief update with its components spread over several CTAs per chunk.

The batched update keeps one CTA per chunk and takes the same steps in the same
order per component, so the two must agree bit for bit.
"""
import numpy as np
import pytest
import torch

import paper_2603_01122_gb300 as pm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("G,B", [(1, 1), (8, 4), (11, 3), (13, 5), (16, 16)])  # 1, 32, 33, 65, 256 components
@pytest.mark.parametrize("n_obs,moving", [(1, True), (64, True), (65, True), (7, False)])
@pytest.mark.parametrize("speeds", [None, (0.5, 1.0)])
def test_groups_equal_one_cta(G, B, n_obs, moving, speeds):
    rng = np.random.default_rng(G * B + n_obs)
    J, n = G * B, 2
    goals = torch.tensor(rng.uniform(0, 8, (G, 2)).astype(np.float32)).cuda()
    beta = torch.tensor((10.0 ** rng.uniform(-2, 2, B)).astype(np.float32)).cuda()
    step = rng.normal(0.0, 0.05, (n_obs, 2)) if moving else np.zeros((n_obs, 2))
    obs = torch.tensor((3.0 + np.concatenate([np.zeros((1, 2)), np.cumsum(step, 0)])).astype(np.float32)).cuda()
    prior = np.log(rng.dirichlet(np.ones(J))).astype(np.float32)
    if J > 2:
        prior[J // 2] = -np.inf
    ctx = pm.pm_create(0)
    try:
        model = pm.make_model(20, 1.0, 0.05, goals, beta, speeds=speeds)
        one, two = torch.tensor(prior).cuda(), torch.tensor(prior).cuda()
        for _ in range(n):  # twice: the tickets are back at zero
            pm.pm_update_posterior(ctx, model, obs, n_obs, one)
        batch = pm.pm_batch_create(ctx, model, 1)
        counts, oob = torch.empty((1, 1, 1), dtype=torch.int32).cuda(), torch.empty(1, dtype=torch.int32).cuda()
        pm.pm_batch_set(batch, [pm.make_human(goals, beta, two, obs[-1], 1, 1, pm.make_grid(0.0, 0.0, 1.0, 1, 1), 1, 1,
                                              counts[0], oob, obs_xy=obs, n_obs=n_obs)])
        for _ in range(n):
            pm.pm_batch_update_posterior(batch)
        pm.pm_sync_status(ctx)
        assert np.array_equal(one.cpu().numpy(), two.cpu().numpy())
        pm.pm_batch_destroy(batch)
    finally:
        pm.pm_destroy(ctx)


def test_scratch_of_a_long_history_serves_many_components_in_a_capture():
    """64 chunks of 4 components need as many partial sums as one chunk of 256:
    after the first call the second one allocates nothing, so it can be captured,
    and the first one's graph stays valid."""
    rng = np.random.default_rng(3)
    beta = torch.tensor((10.0 ** rng.uniform(-1, 1, 16)).astype(np.float32)).cuda()
    goals = torch.tensor(rng.uniform(0, 8, (16, 2)).astype(np.float32)).cuda()
    obs = torch.tensor((3.0 + np.cumsum(rng.normal(0.0, 0.05, (65, 2)), 0)).astype(np.float32)).cuda()

    def calls(G, B, n_obs):
        held = goals[:G].contiguous(), beta[:B].contiguous()
        model = pm.make_model(20, 1.0, 0.05, *held)
        prior = torch.full((G * B,), float(-np.log(G * B))).cuda()
        post = torch.empty_like(prior)
        return post, held, lambda ctx: pm.pm_update_posterior_into(ctx, model, obs, n_obs, prior, post,
                                                                   torch.cuda.current_stream())

    few, many = calls(2, 2, 64), calls(16, 16, 1)
    wants = []
    for post, _, f in (few, many):
        ctx = pm.pm_create(0)
        f(ctx)
        pm.pm_sync_status(ctx)
        wants.append(post.clone())
        pm.pm_destroy(ctx)
    ctx = pm.pm_create(0)
    try:
        few[2](ctx)
        torch.cuda.synchronize()
        graphs = []
        for post, _, f in (few, many):
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                f(ctx)
            graphs.append(g)
        for g, (post, _, _), want in zip(graphs, (few, many), wants):
            post.zero_()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(post, want)
    finally:
        pm.pm_destroy(ctx)
