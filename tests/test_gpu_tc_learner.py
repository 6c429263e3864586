"""The learner's tensor-core passes (CTAs of whole 128-sample tiles) at the edges of their range:
one to four tiles, every hidden width, narrow and full inputs, clusters, every critic layout;
against the FP64 oracle with the tolerances of the other update tests."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import assert_close, cpu, f64
from test_gpu_learner import NETS, check_update, make_run, oracle_buffer, oracle_learner

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hidden,batch,cluster,layout,n_hist",
                         [(32, 128, 1, 0, 16), (32, 384, 1, 2, 0), (64, 512, 2, 1, 16), (64, 128, 1, 3, 1),
                          (128, 128, 1, 1, 16), (128, 384, 1, 0, 8), (128, 512, 4, 3, 0)])
def test_tile_update_parity(gpu, hidden, batch, cluster, layout, n_hist):
    q = gpu
    d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=cluster, layout=layout, n_hist=n_hist)
    try:
        ai = q.ac_info_get(a)
        g = torch.Generator(device="cuda").manual_seed(5)
        for k in ("actor_t", "c1_t", "c2_t"):
            ai[k] += 0.02 * torch.randn(ai[k].shape, device="cuda", generator=g)
        torch.cuda.synchronize()
        for call in range(3):
            info = q.qsim_info_get(h)
            buf = oracle_buffer(info, info["n_envs"])
            L = oracle_learner(q.ac_info_get(a))
            q.ac_update(a, h, 1)
            torch.cuda.synchronize()
            dg = O.td3_update(d, hp, L, buf)
            ai = q.ac_info_get(a)
            check_update(ai, L, dg, hp, f"update{call}")
            assert_close(f64(ai["stats"])[0], dg["critic_loss"], 1.0, what="critic loss")
    finally:
        q.ac_destroy(a)
        q.qsim_destroy(h)


@pytest.mark.parametrize("hidden,batch,cluster", [(32, 128, 1), (64, 256, 2), (128, 256, 1), (128, 512, 4)])
def test_wait_that_runs_out_leaves_the_networks_alone(gpu, hidden, batch, cluster):
    """A one-poll limit on the env set: qsim_sync reports QSIM_ETIMEOUT, no weight, target or
    moment has changed, the counters stand where a full call leaves them, and with the
    default limit the next updates match the oracle."""
    q = gpu
    d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=cluster)
    try:
        q.ac_update(a, h, 2)
        q.qsim_sync(h)
        before = {k: cpu(q.ac_info_get(a)[k]).view(np.uint32).copy() for k in NETS}
        q.qsim_set_wait_limit(h, 1)
        q.ac_update(a, h, 3)
        with pytest.raises(q.QsimError) as ei:
            q.qsim_sync(h)
        assert ei.value.status == -4
        ai = q.ac_info_get(a)
        for k in NETS:
            assert np.array_equal(cpu(ai[k]).view(np.uint32), before[k]), k
        assert (ai["updates"], ai["t_critic"], ai["t_actor"]) == (5, 5, 2)
        q.qsim_set_wait_limit(h, 0)
        for call in range(2):
            info = q.qsim_info_get(h)
            L = oracle_learner(q.ac_info_get(a))
            q.ac_update(a, h, 1)
            q.qsim_sync(h)
            dg = O.td3_update(d, hp, L, oracle_buffer(info, info["n_envs"]))
            check_update(q.ac_info_get(a), L, dg, hp, f"update{call}")
    finally:
        q.ac_destroy(a)
        q.qsim_destroy(h)


def _perturbed(q, a, seed):
    ai = q.ac_info_get(a)
    g = torch.Generator(device="cuda").manual_seed(100 + seed)
    for k in ("actor", "c1", "c2"):
        ai[k] += 0.05 * torch.randn(ai[k].shape, device="cuda", generator=g)
    for k in ("actor_t", "c1_t", "c2_t"):
        ai[k].copy_(ai[k[:-2]])
        ai[k] += 0.02 * torch.randn(ai[k].shape, device="cuda", generator=g)
    return ai


def _w1(ai, k, hidden, inp):
    return ai[k][:hidden * inp].view(hidden, inp)


@pytest.mark.parametrize("small", [1.0, 1e-4])
@pytest.mark.parametrize("hidden,batch,layout", [(32, 128, 0), (64, 256, 1), (128, 128, 0), (128, 256, 2)])
def test_gradients_keep_fp32_accuracy(gpu, hidden, batch, layout, small):
    """The gradient (the first Adam moment after one update from zero) against 64 bits, column
    by column of W1: a column of small inputs (positions and velocities of 1e-4) keeps its
    digits too.  Five products each round their operands to 2^-23 and drop 2^-22 of a
    product, FP32 sums add as much again: 8 x 2^-22."""
    q = gpu
    d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=1, layout=layout)
    try:
        ai = _perturbed(q, a, 0)
        info = q.qsim_info_get(h)
        for rows in (slice(0, 3), slice(7, 13)):
            info["records"][:, rows] *= small
            info["side"][:, rows] *= small
        torch.cuda.synchronize()
        for call in range(2):
            for k in ("m_a", "m_c1", "m_c2"):
                ai[k].zero_()
            torch.cuda.synchronize()
            info = q.qsim_info_get(h)
            buf, L = oracle_buffer(info, info["n_envs"]), oracle_learner(q.ac_info_get(a))
            q.ac_update(a, h, 1)
            torch.cuda.synchronize()
            dg = O.td3_update(d, hp, L, buf)
            ai = q.ac_info_get(a)
            for gk, mk, inp in (("g_c1", "m_c1", info["critic_obs_dim"] + 4), ("g_c2", "m_c2", info["critic_obs_dim"] + 4),
                                ("g_a", "m_a", info["obs_dim"])):
                if gk == "g_a" and not dg["actor_updated"]:
                    continue
                g = dg[gk][:hidden * inp].reshape(hidden, inp)
                e = f64(ai[mk])[:hidden * inp].reshape(hidden, inp) / float(np.float32(1) - np.float32(hp["beta1"])) - g
                rel = np.linalg.norm(e, axis=0) / np.maximum(np.linalg.norm(g, axis=0), 1e-30)
                assert rel.max() < 8 * 2.0**-22, f"update{call}.{mk}: column {rel.argmax()} off by {rel.max():.2e}"
    finally:
        q.ac_destroy(a)
        q.qsim_destroy(h)


@pytest.mark.parametrize("hidden,batch,cluster,layout", [(32, 128, 1, 0), (64, 256, 1, 0), (128, 256, 2, 0), (128, 128, 1, 1)])
def test_values_past_the_half_range(gpu, hidden, batch, cluster, layout):
    """Networks whose first layer is 2^22 times as large and whose second is 2^22 times smaller
    are the same functions: weights and hidden activations past 65,504, or far below it, give
    the oracle's update.  (All networks are set anew for each update: a step of Adam is as
    large for a weight of 1e-8 as for one of 0.1, after which the function is another, and a
    Polyak step puts a share of the large weights into the targets.)"""
    q = gpu
    d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=cluster, layout=layout)
    try:
        ai = _perturbed(q, a, 1)
        info = q.qsim_info_get(h)
        inputs = dict(actor=info["obs_dim"], c1=info["critic_obs_dim"] + 4, c2=info["critic_obs_dim"] + 4)
        orig = {k: ai[k].clone() for k in ("actor", "actor_t", "c1", "c1_t", "c2", "c2_t")}
        for f in (2.0**22, 2.0**-22):
            for call in range(2):
                for k in orig:
                    ai[k].copy_(orig[k])
                for k, inp in inputs.items():
                    n = hidden * inp + hidden
                    ai[k][:n] *= f
                    ai[k][n:n + hidden * hidden] /= f
                    for m in ("m_", "v_"):
                        ai[m + ("a" if k == "actor" else k)].zero_()
                torch.cuda.synchronize()
                L = oracle_learner(q.ac_info_get(a))
                q.ac_update(a, h, 1)
                q.qsim_sync(h)
                dg = O.td3_update(d, hp, L, oracle_buffer(info, info["n_envs"]))
                ai = q.ac_info_get(a)
                for mk, k in (("m_c1", "c1"), ("m_c2", "c2"), ("m_a", "actor")):
                    if k == "actor" and not dg["actor_updated"]:
                        continue
                    got, want, n = f64(ai[mk]), L[mk], hidden * inputs[k]
                    for what, part in (("W1", slice(0, n)), ("rest", slice(n, None))):
                        err = np.linalg.norm((got - want)[part]) / np.linalg.norm(want[part])
                        assert err < 1e-4, f"x{f} update{call}.{mk}.{what}: {err:.2e}"
    finally:
        q.ac_destroy(a)
        q.qsim_destroy(h)


@pytest.mark.parametrize("hidden,batch,cluster", [(32, 128, 1), (64, 256, 2), (128, 128, 1), (128, 512, 4)])
def test_weights_that_outgrow_their_scale_within_a_launch(gpu, hidden, batch, cluster):
    """With a learning rate of 1 the first step makes every network ten times as large, past its
    image's range: two updates in one launch make the image again and give the bits of two
    launches, which always make it."""
    q = gpu
    outs = []
    for calls in ((2, 2), (1, 1, 1, 1)):
        d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=cluster)
        q.ac_destroy(a)
        a = q.ac_create(q.make_ac_config({**hp, "lr": 1.0}, cluster=cluster), h)
        try:
            # (two updates from fresh weights, twice)
            ai = q.ac_info_get(a)
            start = {k: ai[k].clone() for k in NETS}
            for i, n in enumerate(calls):
                if i == len(calls) // 2:
                    q.qsim_sync(h)
                    outs.append([cpu(ai[k]).view(np.uint32).copy() for k in NETS])
                    for k in NETS:
                        ai[k].copy_(start[k])
                    torch.cuda.synchronize()
                q.ac_update(a, h, n)
            q.qsim_sync(h)
            outs.append([cpu(ai[k]).view(np.uint32).copy() for k in NETS])
            assert all(np.isfinite(cpu(ai[k])).all() for k in NETS)
        finally:
            q.ac_destroy(a)
            q.qsim_destroy(h)
    for x, y in zip(outs[0] + outs[1], outs[2] + outs[3]):
        assert np.array_equal(x, y)


def test_regression_settles_every_unit_near_zero_in_fp32_order(gpu):
    """Hidden 128: one large weight in each layer of the critics, on paths the output does not
    see (unit 0's second-layer column and its output weight are zero), widens the band around
    zero so far that thousands of units of every row are formed in FP32 order, by thread in
    layer 1 and by warp in layer 2; the update is the oracle's."""
    q = gpu
    hidden, batch = 128, 256
    d, h, a, hp = make_run(q, hidden=hidden, batch=batch, cluster=1)
    try:
        ai = _perturbed(q, a, 2)
        info = q.qsim_info_get(h)
        inp = info["critic_obs_dim"] + 4
        for k in ("c1", "c2"):
            _w1(ai, k, hidden, inp)[0, 5] = 2.0e3
            n = hidden * inp + hidden
            w2 = ai[k][n:n + hidden * hidden].view(hidden, hidden)
            w2[:, 0] = 0.0
            w2[0, 7] = 2.0e3
            ai[k][n + hidden * hidden + hidden] = 0.0  # W3's entry of unit 0
        torch.cuda.synchronize()
        for call in range(2):
            info = q.qsim_info_get(h)
            L = oracle_learner(q.ac_info_get(a))
            q.ac_update(a, h, 1)
            q.qsim_sync(h)
            dg = O.td3_update(d, hp, L, oracle_buffer(info, info["n_envs"]))
            check_update(q.ac_info_get(a), L, dg, hp, f"update{call}")
    finally:
        q.ac_destroy(a)
        q.qsim_destroy(h)
