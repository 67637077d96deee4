"""Differentiable SPaSM costs for PyTorch (torch.autograd.Function around the CUDA kernels).

``traj_cost(problem, q, lam, mu)`` is the stage-2 augmented-Lagrangian objective of each
trajectory particle (Sec. III-B; cost terms of the appendix) and ``place_cost(problem, x,
quadratic)`` the stage-1 tower placement cost (appendix, Alg. 1's linear / quadratic forms).
A forward pass whose input needs a gradient runs the evaluation kernel once with its analytic
backward, which shares the kinematics, the culls and the residuals with the cost, and keeps the
gradient (the size of the input; no transforms are stored); the backward pass scales it by the
incoming gradient, particle by particle.  A second kernel run in the backward pass, with
everything computed again, took 2.36 ms in place of 1.29 ms for 4096 trajectories of the
10-block tower.  Without a gradient to compute the forward pass runs the kernel without its backward part;
a caller who wants only the value of an input that requires a gradient says so with torch.no_grad()
(without it the call holds a tensor of the input's size and takes 1.15 in place of 1.06 ms there, 38 in
place of 28 us for a few placements).
Inputs are CUDA float32 tensors; no computation happens in Python.
"""
from __future__ import annotations

import torch

from . import spasm as S


def _pad8(q: torch.Tensor, C: int) -> torch.Tensor:
    if q.dim() != 3 or q.shape[1] != C or q.shape[2] not in (7, 8):
        raise ValueError(f"q must be (n, {C}, 7|8)")
    if q.shape[2] == 8:
        return q.detach().contiguous().float()
    out = torch.zeros(q.shape[0], C, 8, device=q.device, dtype=torch.float32)
    out[:, :, :7] = q.detach()
    return out


class TrajCost(torch.autograd.Function):
    @staticmethod
    def forward(ctx, q, problem, lam, mu, recording=True):   # recording: a backward pass can follow
        qq = _pad8(q, problem.C)
        n = qq.shape[0]
        L = torch.empty(n, device=q.device, dtype=torch.float32)
        lam_c = None if lam is None else lam.detach().contiguous().float()
        mu_c = None if mu is None else mu.detach().contiguous().float()
        grad = torch.empty_like(qq) if recording and ctx.needs_input_grad[0] else None
        S.spasm_traj_eval(problem, n, qq, lam_c, mu_c, L, grad)
        ctx.width = q.shape[2]
        if grad is not None:
            # qq beside it: an input changed in place before the backward pass is reported
            ctx.save_for_backward(qq, grad, *(t for t in (lam_c, mu_c) if t is not None))
        return L

    @staticmethod
    def backward(ctx, gL):
        grad = ctx.saved_tensors[1]
        g = grad[:, :, : ctx.width] * gL.to(grad.dtype)[:, None, None]
        return g, None, None, None, None


class PlaceCost(torch.autograd.Function):
    @staticmethod
    def forward(ctx, x, problem, quadratic, recording=True):
        xx = x.detach().contiguous().float()   # (4B, n) structure of arrays
        n = xx.shape[1]
        cost = torch.empty(n, device=x.device, dtype=torch.float32)
        grad = torch.empty_like(xx) if recording and ctx.needs_input_grad[0] else None
        S.spasm_place_eval(problem, n, xx, int(quadratic), cost, grad)
        if grad is not None:
            ctx.save_for_backward(xx, grad)
        return cost

    @staticmethod
    def backward(ctx, gc):
        grad = ctx.saved_tensors[1]
        return grad * gc.to(grad.dtype)[None, :], None, None, None


def traj_cost(problem, q, lam=None, mu=None):
    """Per-particle stage-2 objective L(q) (n,), differentiable w.r.t. q (n, C, 7|8)."""
    return TrajCost.apply(q, problem, lam, mu, torch.is_grad_enabled())


def place_cost(problem, x, quadratic: bool = False):
    """Per-particle stage-1 placement cost (n,), differentiable w.r.t. x (4B, n)."""
    return PlaceCost.apply(x, problem, quadratic, torch.is_grad_enabled())
