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
