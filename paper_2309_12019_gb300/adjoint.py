"""Gradients of a final-time misfit with respect to the initial DOFs, through the
library's discrete adjoint (dgw_adjoint_step), as torch.autograd.Functions.

rollout(ctx, U0, dt, nsteps, every) advances U0 by nsteps SSP-RK3 steps and keeps a
checkpoint every `every` steps; its backward pass recomputes each segment from its
checkpoint, keeping every step's state and its two stage states (dgw_rk_step_stages),
and runs dgw_adjoint_step_stages through the segment in reverse, so that no stage is
evaluated twice in the backward pass.  The last segment, with which the backward pass
begins, is kept by the forward pass when a gradient is asked for, so that its states are
not recomputed.  A context holds one such segment at most, that of its latest rollout: an
earlier one, of a graph that was chained or is still waiting for its backward pass, falls
back to its checkpoint.  So the largest memory in use, the checkpoints and one segment, is
that of a backward pass which recomputes every segment; it is held from the forward pass on.
misfit(ctx, U, U_target) is J = 1/2 int (U_h - U_target)^2 with dJ/dU from dgw_misfit.
All arithmetic runs in the library's kernels; this module only orders the calls.
"""
from __future__ import annotations

import weakref

import torch


class _Kept:
    """The stages of a rollout's last segment, until its backward pass takes them or the next
    rollout on the context drops them."""

    def __init__(self, dctx, steps):
        self.steps = steps
        dctx.kept_segment = weakref.ref(self)

    def take(self):
        steps, self.steps = self.steps, None
        return steps

    @staticmethod
    def drop(dctx):
        kept = getattr(dctx, "kept_segment", lambda: None)()
        if kept is not None:
            kept.take()


def _segment(dctx, U, dt, n, last_state):
    """n steps from U keeping every step's (U_n, U_1, U_2); and the state after them, None
    unless last_state (the last step's third stage is then skipped)."""
    steps = []
    for i in range(n):
        U1, U2 = torch.empty_like(U), torch.empty_like(U)
        nxt = torch.empty_like(U) if last_state or i < n - 1 else None
        dctx.rk_step_stages(U, dt, U1, U2, nxt)
        steps.append((U, U1, U2))
        U = nxt
    return steps, U


class _Rollout(torch.autograd.Function):
    @staticmethod
    def forward(ctx_, U0, dctx, dt, nsteps, every, grad):
        U = U0.detach().clone().contiguous()
        # (what has no adjoint has no stage states either: its forward pass takes plain steps)
        keep = grad and dctx.problem.rk_order == 3 and "state" not in dctx.problem.bc
        checkpoints, last, done = [], None, 0
        while done < nsteps:
            n = min(every, nsteps - done)
            done += n
            if keep and done == nsteps:
                _Kept.drop(dctx)
                checkpoints.append(U)
                steps, U = _segment(dctx, U, dt, n, True)
                last = _Kept(dctx, steps)
            else:
                checkpoints.append(U.clone())
                dctx.rk_step(U, dt, n)
        ctx_.dctx, ctx_.dt, ctx_.nsteps, ctx_.every = dctx, dt, nsteps, every
        ctx_.checkpoints, ctx_.last = checkpoints, last
        return U

    @staticmethod
    def backward(ctx_, gout):
        dctx, dt, nsteps, every = ctx_.dctx, ctx_.dt, ctx_.nsteps, ctx_.every
        lam = gout.detach().clone().contiguous()
        for seg in reversed(range(len(ctx_.checkpoints))):
            steps = ctx_.last.take() if ctx_.last is not None else None
            ctx_.last = None
            if steps is None:
                steps, _ = _segment(dctx, ctx_.checkpoints[seg], dt, min(every, nsteps - seg * every), False)
            while steps:
                Un, U1, U2 = steps.pop()
                dctx.adjoint_step_stages(Un, U1, U2, lam, lam, dt)
        ctx_.checkpoints = None
        return lam, None, None, None, None, None


class _Misfit(torch.autograd.Function):
    @staticmethod
    def forward(ctx_, U, U_target, dctx):
        grad = torch.empty_like(U)
        J = dctx.misfit(U.contiguous(), U_target.contiguous(), grad)
        ctx_.save_for_backward(grad)
        return torch.tensor(J, dtype=torch.float64, device=U.device)

    @staticmethod
    def backward(ctx_, gJ):
        (grad,) = ctx_.saved_tensors
        return grad * gJ.to(grad.dtype), None, None


def rollout(dctx, U0, dt: float, nsteps: int, every: int = 20):
    # (inside forward() gradients are off, and needs_input_grad ignores no_grad)
    grad = U0.requires_grad and torch.is_grad_enabled()
    return _Rollout.apply(U0, dctx, float(dt), int(nsteps), int(every), grad)


def misfit(dctx, U, U_target):
    return _Misfit.apply(U, U_target, dctx)
