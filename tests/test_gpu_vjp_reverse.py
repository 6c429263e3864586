"""The reverse sweep on a workspace that a forward-only call filled gives the gradients of the
call that runs both, bit for bit, and can be repeated."""
import numpy as np
import pytest
import torch

import workloads as W
from helpers import cpu
from paper_2311_13081_gb300 import diff

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,hidden,n,H,ckpt", [(0, 64, 64, 23, 10), (0, 64, 4, 1, 5), (1, 64, 68, 23, 10),
                                                  (1, 32, 4, 7, 20), (1, 16, 32, 9, 4)])
def test_reverse_alone_equals_both(gpu, mode, hidden, n, H, ckpt):
    q = gpu
    g = torch.Generator("cuda").manual_seed(n + H)
    veh = q.make_params(W.VEHICLE)
    s0 = torch.tensor(W.random_states(3, n).T.copy(), dtype=torch.float32, device="cuda")
    prm = torch.tensor(W.random_params(4, n).T.copy(), dtype=torch.float32, device="cuda")
    acts = torch.rand(H, 4, n, device="cuda", generator=g) * 2 - 1
    actor = torch.randn(q.param_count(82, hidden, 4), device="cuda", generator=g) * 0.1
    seed = torch.rand(n, device="cuda", generator=g)
    desc = diff.make_desc(n, n, H, ckpt, mode, (1.0, 0.5, 0.2, 0.05), hidden=hidden)
    a, p = (acts, None) if mode == 0 else (None, actor)

    def grads():
        return (torch.zeros_like(acts) if mode == 0 else None, torch.zeros_like(actor) if mode else None,
                torch.zeros(4, n, device="cuda"))

    ws = [torch.empty(q.qsim_vjp_workspace(desc) // 4 + 4, device="cuda") for _ in range(2)]
    loss = torch.zeros(n, device="cuda")
    want = grads()
    q.qsim_rollout_vjp(desc, veh, s0, prm, a, p, seed, loss, *want, None, ws[0])
    q.qsim_rollout_vjp(desc, veh, s0, prm, a, p, None, loss, None, None, None, None, ws[1])
    for _ in range(2):
        got = grads()
        q.qsim_rollout_vjp_reverse(desc, veh, s0, prm, a, p, seed, *got, ws[1])
        torch.cuda.synchronize()
        for x, y in zip(got, want):
            if x is not None:
                assert np.array_equal(cpu(x).view(np.uint32), cpu(y).view(np.uint32))


def _autograd_inputs(q, n, H, closed, hidden=64):
    g = torch.Generator("cuda").manual_seed(n + H)
    veh = q.make_params(W.VEHICLE)
    s0 = torch.tensor(W.random_states(3, n).T.copy(), dtype=torch.float32, device="cuda")
    prm = torch.tensor(W.random_params(4, n).T.copy(), dtype=torch.float32, device="cuda").requires_grad_()
    x = (torch.randn(q.param_count(82, hidden, 4), device="cuda", generator=g) * 0.1 if closed
         else torch.rand(H, 4, n, device="cuda", generator=g) * 2 - 1).requires_grad_()
    desc = diff.make_desc(n, n, H, 10, int(closed), (1.0, 0.5, 0.2, 0.05), hidden=hidden)
    return veh, s0, prm, x, desc


@pytest.mark.parametrize("closed", [False, True])
def test_structs_changed_after_the_forward_pass(gpu, closed):
    """The backward pass belongs to the loss that was computed: the caller's descriptor and
    vehicle may be reused for something else in between."""
    q = gpu
    veh, s0, prm, x, desc = _autograd_inputs(q, 68, 23, closed)
    want = torch.autograd.grad(diff.RolloutLoss.apply(prm, x, s0, veh, desc).sum(), (prm, x))
    loss = diff.RolloutLoss.apply(prm, x, s0, veh, desc)
    desc.w_p, desc.w_q, veh.kf = 7.0, 0.0, 2.0 * veh.kf
    got = torch.autograd.grad(loss.sum(), (prm, x))
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("closed,hidden", [(False, 64), (True, 64), (True, 16)])
def test_pending_losses_hold_their_rollouts_only(gpu, closed, hidden):
    """Two pending losses and a retained graph give the gradients of one loss at a time, bit
    for bit, and a pending loss holds its checkpoints, actions and loss row, no scratch."""
    q = gpu
    veh, s0, prm, x, desc = _autograd_inputs(q, 132, 23, closed, hidden)
    x2 = (x.detach() * 0.5).requires_grad_()
    want = [torch.autograd.grad(diff.RolloutLoss.apply(prm, v, s0, veh, desc).sum(), (prm, v)) for v in (x, x2)]
    torch.cuda.synchronize()
    before = torch.cuda.memory_allocated()
    losses = [diff.RolloutLoss.apply(prm, v, s0, veh, desc) for v in (x, x2)]
    held = (torch.cuda.memory_allocated() - before) // 2
    rollout = 4 * desc.ld * (-(-desc.H // desc.ckpt) * 17 + 4 * desc.H)  # checkpoints and actions
    assert held <= rollout + 4 * desc.ld + 4 * 512, (held, rollout, q.qsim_vjp_workspace(desc))
    for loss, v, w in ((losses[1], x2, want[1]), (losses[0], x, want[0]), (losses[1], x2, want[1])):
        for a, b in zip(torch.autograd.grad(loss.sum(), (prm, v), retain_graph=True), w):
            assert torch.equal(a, b)


def test_workspace_parts_too_small_are_refused(gpu):
    q = gpu
    veh, s0, prm, x, desc = _autograd_inputs(q, 64, 23, True)
    kept = torch.empty(q.qsim_vjp_kept(desc) // 4, device="cuda")
    scratch = torch.empty((q.qsim_vjp_workspace(desc) - q.qsim_vjp_kept(desc)) // 4, device="cuda")
    loss, gx = torch.zeros(64, device="cuda"), torch.zeros_like(x)
    q.qsim_rollout_vjp_keep(desc, veh, s0, prm, None, x, loss, None, kept, scratch)
    desc.H += 40
    for k, s in ((kept, torch.empty(1 << 24, device="cuda")), (torch.empty(1 << 22, device="cuda"), scratch[:100])):
        with pytest.raises(q.QsimError, match="workspace parts"):
            q.qsim_rollout_vjp_from(desc, veh, s0, prm, None, x, None, None, gx, None, k, s)
