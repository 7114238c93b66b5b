"""Differentiable no-flow rollout of the coupled surfactant step.

SurfactantRollout is a torch.autograd.Function: its forward runs `nsteps`
steps of the App. C step from f0 = Gamma0 delta_phi (Sec. 2.3) and returns
the loss L = sum_c V_c |F_Ma,c|^2 of the final Marangoni force; its backward
is the hand-written discrete adjoint of the library (sfx_adjoint_step,
sfx_marangoni_loss, sfx_f_from_gamma), giving dL/dGamma0 and dL/dtheta for
theta = (k_a, k_d, D_f, D_F).  The forward keeps a checkpoint of the state
every K steps and every state of the last segment, which the backward walks
first, freeing each state behind its step (a second backward of a retained
graph recomputes them); the backward recomputes each earlier segment of K steps
from its checkpoint and walks it in the same way.  An open graph so holds its
checkpoints and the states of at most K steps, and its backward never more than
that.  (Recomputing the last segment, once for its end and once for its states,
ran every step of a rollout within K steps three times: eight steps at 256x256
with their gradient 7.65 -> 4.4 ms.)  The forward may run in an SFX_F32
context (double-float state); the adjoint always works in FP64 on these
states.  Every step of the computation runs in libsfx kernels.
"""
from __future__ import annotations

import dataclasses
from typing import Optional

import torch

from ._lib import SFX_F32, SFX_F64, Params


@dataclasses.dataclass
class RolloutSetup:
    """Everything of the rollout that is not differentiated."""
    context: object            # Context of the grid (SFX_F64 or SFX_F32)
    params: object             # base sfx_params-like object (theta overrides 4 fields)
    phi: torch.Tensor          # double phase field
    C: torch.Tensor            # VoF fraction (double) for delta_m
    F0: torch.Tensor           # initial bulk concentration (double)
    dt: float
    nsteps: int
    K: int = 20                # checkpoint interval
    tol: float = 1e-12         # forward solve tolerance
    adj_tol: float = 1e-13     # adjoint solve tolerance
    dm_mode: int = 1
    opts: Optional[object] = None

    def params_with(self, theta):
        from . import params_struct
        ps = params_struct(self.params)
        ps.ka, ps.kd, ps.Df, ps.DF = (float(v) for v in theta)
        return ps


def _forward_steps(setup: RolloutSetup, ps: Params, f, F, n):
    """n steps from (f, F) in the context's state layout, in place."""
    from . import default_opts
    ctx = setup.context
    o = setup.opts if setup.opts is not None else default_opts(tol=setup.tol, max_cycles=400)
    for _ in range(n):
        # no stats: the step then skips its totals and their host wait (a
        # step that fails to converge still raises)
        ctx.sfx_surfactant_step(ps, setup.phi, f, F, setup.dt, opts=o, stats=False)


def _segment(setup: RolloutSetup, ps: Params, start, n):
    """The states after each of n steps from the checkpoint `start`."""
    f, F = (t.clone() for t in start)
    states = []
    for _ in range(n):
        _forward_steps(setup, ps, f, F, 1)
        states.append((f.clone(), F.clone()))
    return states


def _to_state(ctx, x):
    return ctx.sfx_df_pack(x) if ctx.precision == SFX_F32 else x.clone()


def _to_double(ctx, x):
    return ctx.sfx_df_unpack(x) if ctx.precision == SFX_F32 else x


class SurfactantRollout(torch.autograd.Function):
    """loss = SurfactantRollout.apply(gamma0, theta, setup)."""

    @staticmethod
    def forward(fctx, gamma0, theta, setup: RolloutSetup):
        ctx = setup.context
        ps = setup.params_with(theta.detach().cpu().tolist())
        f0 = ctx.sfx_f_from_gamma(gamma0.detach().contiguous(), setup.phi, ps.eps)
        f, F = _to_state(ctx, f0), _to_state(ctx, setup.F0)
        checkpoints = [(f.clone(), F.clone())]
        done = 0
        while setup.nsteps - done > setup.K:
            _forward_steps(setup, ps, f, F, setup.K)
            done += setup.K
            checkpoints.append((f.clone(), F.clone()))
        last = []
        for _ in range(setup.nsteps - done):
            _forward_steps(setup, ps, f, F, 1)
            if any(fctx.needs_input_grad):
                last.append((f.clone(), F.clone()))
        L, _ = ctx.sfx_marangoni_loss(ps, _to_double(ctx, f), setup.phi, setup.C, setup.dm_mode,
                                      grad=False)
        fctx.setup = setup
        fctx.ps = ps
        fctx.checkpoints = checkpoints
        fctx.last = last
        fctx.theta_device = theta.device
        fctx.theta_dtype = theta.dtype
        return torch.tensor(L, dtype=torch.float64)

    @staticmethod
    def backward(fctx, gL):
        from . import default_opts
        setup, ps = fctx.setup, fctx.ps
        ctx = setup.context
        o = default_opts(tol=setup.adj_tol, max_cycles=1000, nu1=10, nu2=10)
        last, fctx.last = fctx.last, None
        if last is None:           # a second backward of the same graph
            last = _segment(setup, ps, fctx.checkpoints[-1],
                            setup.nsteps - (len(fctx.checkpoints) - 1) * setup.K)
        # the final state, for dL/df
        last_f = (last or fctx.checkpoints)[-1][0]
        _, gf = ctx.sfx_marangoni_loss(ps, _to_double(ctx, last_f), setup.phi, setup.C,
                                       setup.dm_mode, grad=True)
        lam_f = gf * float(gL)
        lam_F = torch.zeros_like(lam_f)
        dtheta = [0.0, 0.0, 0.0, 0.0]
        for s in range(len(fctx.checkpoints) - 1, -1, -1):
            states = last if s == len(fctx.checkpoints) - 1 else \
                _segment(setup, ps, fctx.checkpoints[s], setup.K)
            while states:          # (frees each state behind its step)
                f1, F1 = states.pop()
                ctx.sfx_adjoint_step(ps, setup.phi, _to_double(ctx, f1), _to_double(ctx, F1),
                                     setup.dt, lam_f, lam_F, dtheta, o)
        dgamma = ctx.sfx_f_from_gamma(lam_f, setup.phi, ps.eps)
        dth = torch.tensor(dtheta, dtype=fctx.theta_dtype, device=fctx.theta_device)
        return dgamma, dth, None
