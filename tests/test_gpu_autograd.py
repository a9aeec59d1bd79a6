"""The autograd function's contract: which inputs may ask for a gradient, what is refused, what a value costs."""
import numpy as np
import pytest
import torch

import paper_2603_01122_gb300 as pm
from gpu_util import dev
from paper_2603_01122_gb300 import autograd
from paper_2603_01122_gb300.autograd import MarginalLogLik, marginal_loglik

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = pm.pm_create(0)
    yield c
    pm.pm_destroy(c)


def _inputs():
    """Two short walks, G = 2, B = 3: goals, speed, w, beta, offsets, traj, log_prior."""
    rng = np.random.default_rng(5)
    th = rng.uniform(0.0, 6.28, (2, 9))
    step = 0.1 * np.stack([np.cos(th), np.sin(th)], -1)
    traj = np.concatenate([np.concatenate([[[1.0, 2.0]], [1.0, 2.0] + np.cumsum(s, 0)]) for s in step])
    return dict(goals=dev(rng.uniform(0.0, 5.0, (2, 2))), speed=torch.tensor(1.0).cuda(),
                w=torch.tensor([1.0, 1.0]).cuda(), beta=dev([0.5, 1.0, 4.0]),
                offsets=dev(np.array([0, 10, 20], np.int32), torch.int32), traj=dev(traj),
                log_prior=dev(np.full(6, -np.log(6.0))))


def _call(ctx, p, f=marginal_loglik):
    args = (p["goals"], p["speed"], p["w"], p["beta"], 12, 0.1, p["offsets"], p["traj"], p["log_prior"], ctx)
    return f(*args)


@pytest.mark.parametrize("which", [("beta",), ("traj",), ("log_prior",), ("beta", "goals"), ("w",), ("speed", "traj")])
def test_any_input_may_require_a_gradient(ctx, which):
    """goals, speed and w get theirs; the data get none, alone or beside them."""
    p = _inputs()
    for k in which:
        p[k].requires_grad_()
    L = _call(ctx, p)
    L.backward()
    full = _inputs()
    for k in ("goals", "speed", "w"):
        full[k].requires_grad_()
    L_full = _call(ctx, full)
    L_full.backward()
    assert torch.equal(L, L_full)
    for k in p:
        if k in which and k in ("goals", "speed", "w"):
            assert torch.equal(p[k].grad, full[k].grad)
        else:
            assert p[k].grad is None


@pytest.mark.parametrize("which", ["goals", "beta"])
def test_input_changed_before_backward_is_refused(ctx, which):
    p = _inputs()
    p[which].requires_grad_()
    L = _call(ctx, p)
    p["traj"].add_(1.0)
    with pytest.raises(RuntimeError, match="modified by an inplace operation"):
        L.backward()


@pytest.mark.parametrize("g", [float("inf"), float("nan")])
@pytest.mark.parametrize("which", ["goals", "beta"])
def test_non_finite_gradient_is_refused(ctx, which, g):
    p = _inputs()
    p[which].requires_grad_()
    with pytest.raises(pm.PmError, match="grad_out must be finite") as e:
        (g * _call(ctx, p)).backward()
    assert e.value.status == pm.PM_EINVAL
    assert p[which].grad is None


@pytest.mark.parametrize("call", [marginal_loglik, MarginalLogLik.apply])
@pytest.mark.parametrize("mode", [torch.no_grad, torch.inference_mode])
def test_value_without_grad_mode_takes_no_gradient_pass(ctx, monkeypatch, call, mode):
    p = _inputs()
    for k in ("goals", "speed", "w"):
        p[k].requires_grad_()
    want = _call(ctx, p)

    def refuse(*_):
        raise AssertionError("gradient pass in a value-only call")

    monkeypatch.setattr(autograd, "pm_loglik_value_grad", refuse)
    with mode():
        got = _call(ctx, p, call)
    assert torch.equal(got, want) and not got.requires_grad


@pytest.mark.parametrize("K,speeds", [(12, None), (36, None), (16, (0.5, 1.0, 1.5))])
def test_value_grad_rounds_to_the_scaled_gradient(ctx, K, speeds):
    """The FP64 gradient, scaled and rounded to FP32, is what pm_loglik_backward
    writes, bit for bit; a NULL gradient is refused."""
    p = _inputs()
    model = pm.make_model(K, 1.0, 0.1, p["goals"], p["beta"], w1=0.7, w2=1.3, speeds=speeds)
    args = (ctx, model, 2, p["offsets"], 20, p["traj"], p["log_prior"])
    L, L_b = torch.empty(1).cuda(), torch.empty(1).cuda()
    grad = torch.empty(7, dtype=torch.float64).cuda()
    pm.pm_loglik_value_grad(*args, L, grad)
    for g in (1.0, -2.5, 1e-3, 3.14159274, 1e30):
        dg, dv, dw = torch.empty((2, 2)).cuda(), torch.empty(1).cuda(), torch.empty(2).cuda()
        pm.pm_loglik_backward(*args, g, L_b, dg, dv, dw)
        pm.pm_sync_status(ctx)
        want = torch.cat([dg.ravel(), dv, dw])
        got = (grad * torch.tensor(g, dtype=torch.float32).double().cuda()).float()
        assert torch.equal(L, L_b) and torch.equal(got, want), g
    with pytest.raises(pm.PmError, match="grad is NULL") as e:
        pm.pm_loglik_value_grad(*args, L, None)
    assert e.value.status == pm.PM_EINVAL
