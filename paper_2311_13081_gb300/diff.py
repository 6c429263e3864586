"""torch.autograd wrapper of qsim_rollout_vjp (differentiable H-step quadrotor rollout).

The forward pass and the reverse sweep both run in libqsim; this module only allocates the
workspace with torch and routes ``grad_output`` into the library as the per-env seed.
"""
from __future__ import annotations

import torch

from . import (QsimParams, QsimVjpDesc, _lib, load, qsim_rollout_vjp_from, qsim_rollout_vjp_keep,
               qsim_vjp_kept, qsim_vjp_workspace)


def make_desc(n, ld, H, ckpt, mode, weights, dt=0.01, renorm=1, n_hist=16, hidden=64,
              lanes_per_env=0):
    d = QsimVjpDesc()
    d.n, d.ld, d.H, d.ckpt, d.mode = int(n), int(ld), int(H), int(ckpt), int(mode)
    d.n_hist, d.hidden = int(n_hist), int(hidden)
    d.lanes_per_env = int(lanes_per_env)
    d.w_p, d.w_q, d.w_v, d.w_a = (float(x) for x in weights)
    d.dt, d.renorm = float(dt), int(renorm)
    return d


def _floats(nbytes):
    return torch.empty((nbytes + 3) // 4, dtype=torch.float32, device="cuda")


def _scratch(desc):
    return _floats(qsim_vjp_workspace(desc) - qsim_vjp_kept(desc))


class RolloutLoss(torch.autograd.Function):
    """loss_e of an H-step rollout; differentiable w.r.t. ``params`` rows m, Jx, Jy, Jz
    and w.r.t. ``x`` = actions [H][4][ld] (open loop) or the flat actor (closed loop).

    The forward pass's checkpoints and actions go to the backward pass as a saved tensor,
    which then runs the reverse sweep alone (4,096 envs x 200 open-loop steps: 682 us for
    both passes when the rollout was run again, 546 us now).  The rest of the workspace is
    scratch of either pass and not held in between (closed loop, 4,096 envs x 200 steps,
    checkpoint 20, hidden 64: 16 MB a pending loss, 272 MB with it)."""

    @staticmethod
    def forward(ctx, params, x, s0, veh: QsimParams, desc: QsimVjpDesc):
        load()
        # copies: the structs are the caller's, who may change them before the backward pass
        desc, veh = QsimVjpDesc.from_buffer_copy(desc), QsimParams.from_buffer_copy(veh)
        ld, n = desc.ld, desc.n
        loss = torch.zeros(ld, device="cuda")
        kept = _floats(qsim_vjp_kept(desc))
        acts = x if desc.mode == 0 else None
        actor = x if desc.mode == 1 else None
        qsim_rollout_vjp_keep(desc, veh, s0, params, acts, actor, loss, None, kept, _scratch(desc))
        ctx.save_for_backward(params, x, s0, kept)
        ctx.veh, ctx.desc = veh, desc
        return loss[:n]

    @staticmethod
    def backward(ctx, g_loss):
        params, x, s0, kept = ctx.saved_tensors
        desc, veh = ctx.desc, ctx.veh
        ld, n = desc.ld, desc.n
        seed = torch.zeros(ld, device="cuda")
        seed[:n] = g_loss
        gp = torch.zeros(4, ld, device="cuda")
        gx = torch.zeros_like(x)
        if desc.mode == 0:
            qsim_rollout_vjp_from(desc, veh, s0, params, x, None, seed, gx, None, gp, kept, _scratch(desc))
        else:
            qsim_rollout_vjp_from(desc, veh, s0, params, None, x, seed, None, gx, gp, kept, _scratch(desc))
        g_params = torch.zeros_like(params)
        g_params[0:4] = gp
        return g_params, gx, None, None, None


def rollout_loss(s0, params, veh, H, ckpt, weights, actions=None, actor=None, n_hist=16,
                 hidden=64, dt=0.01, renorm=1):
    """Per-env loss of an H-step rollout from states ``s0`` [17][ld] with per-env
    ``params`` [8][ld]; pass ``actions`` [H][4][ld] (open loop) or a flat ``actor``."""
    ld = s0.shape[1]
    n = ld if not hasattr(s0, "n_envs") else s0.n_envs
    mode = 0 if actions is not None else 1
    desc = make_desc(n, ld, H, ckpt, mode, weights, dt, renorm, n_hist, hidden)
    return RolloutLoss.apply(params, actions if mode == 0 else actor, s0, veh, desc)
