"""torch.autograd.Function over the library's log-likelihood adjoint.

``MarginalLogLik.apply(goals, speed, w, beta, K, dt, offsets, traj, log_prior, ctx, speeds, snap_heading)``
returns the marginal log-likelihood L of the observed trajectories (a CUDA
scalar). Where a gradient is wanted (an input requires one and the grad mode is
on), the forward call takes L and the gradient with respect to the goal
coordinates, the speed and the Q weights from one pass of the adjoint kernel (it
forms both from the same weights; a second pass in backward cost as much again),
and backward scales it on the device, in FP64 before the rounding to FP32. An
incoming gradient that is not finite is refused (PM_EINVAL), as
pm_loglik_backward refuses it. ``speed`` and ``w`` are read to the host once per
call (the C ABI takes them as scalars), the incoming gradient once in backward.
``speeds`` (a tuple of multipliers, or None for one speed) selects the control
set of several speeds; ``snap_heading`` reads each observed heading as the
nearest enabled heading. 256 trajectories, G = 4, B = 10, value and gradient
waited for: 440 -> 357 us, a value alone 152.
"""
from __future__ import annotations

import math

import torch

from . import PM_EINVAL, PmError, make_model, pm_loglik_forward, pm_loglik_value_grad


def _call(goals, speed, w, beta, K, dt, offsets, traj, log_prior, ctx, speeds=None, snap_heading=False):
    """Arguments of the library's log-likelihood calls up to L (the last one), and their stream."""
    v = float(speed.detach().reshape(()).item())
    w1, w2 = w.detach().reshape(2).tolist()
    goals = goals.detach().contiguous()
    model = make_model(K, v, dt, goals, beta, w1=w1, w2=w2, speeds=speeds, snap_heading=snap_heading)
    out = torch.empty((), dtype=torch.float32, device=goals.device)
    stream = torch.cuda.current_stream(goals.device)
    return (ctx, model, offsets.numel() - 1, offsets, traj.shape[0], traj, log_prior, out), goals, stream


class _Value(torch.autograd.Function):
    """L alone, for calls with the grad mode off (no backward)."""

    @staticmethod
    def forward(fctx, *inputs):
        args, _, stream = _call(*inputs)
        pm_loglik_forward(*args, stream)
        return args[-1]


class MarginalLogLik(torch.autograd.Function):
    @classmethod
    def apply(cls, *args):
        # needs_input_grad is about the inputs alone, whatever the grad mode,
        # and forward always runs with it off: a value-only call is seen here
        return super().apply(*args) if torch.is_grad_enabled() else _Value.apply(*args)

    @staticmethod
    def forward(fctx, goals, speed, w, beta, K, dt, offsets, traj, log_prior, *options):
        args, goals_c, stream = _call(goals, speed, w, beta, K, dt, offsets, traj, log_prior, *options)
        if any(fctx.needs_input_grad[:3]):
            grad = torch.empty(goals_c.numel() + 3, dtype=torch.float64, device=goals.device)
            pm_loglik_value_grad(*args, grad, stream)
        else:
            grad = None  # backward may still run, for beta, traj or log_prior: they get no gradient
            pm_loglik_forward(*args, stream)
        # the inputs too: a change to them before backward is refused, as ever
        fctx.save_for_backward(grad, goals_c, speed, w, beta, offsets, traj, log_prior)
        return args[-1]

    @staticmethod
    def backward(fctx, grad_out):
        grad, goals, speed, w = fctx.saved_tensors[:4]
        g = grad_out.item()  # one read; it also makes the scaling by 1 of a plain backward() unnecessary
        if not math.isfinite(g):
            raise PmError(PM_EINVAL, "grad_out must be finite")
        out = [None] * len(fctx.needs_input_grad)
        if grad is not None:
            d = (grad if g == 1.0 else grad * g).to(torch.float32)  # the product in FP64
            n = goals.numel()
            need = fctx.needs_input_grad
            if need[0]:
                out[0] = d[:n].view(goals.shape)
            if need[1]:
                out[1] = d[n:n + 1].to(speed.device).reshape(speed.shape)
            if need[2]:
                out[2] = d[n + 1:].to(w.device).reshape(w.shape)
        return tuple(out)


def marginal_loglik(goals, speed, w, beta, K, dt, offsets, traj, log_prior, ctx, speeds=None, snap_heading=False):
    """Differentiable marginal log-likelihood (see MarginalLogLik)."""
    return MarginalLogLik.apply(goals, speed, w, beta, K, dt, offsets, traj, log_prior, ctx,
                                None if speeds is None else tuple(speeds), bool(snap_heading))
