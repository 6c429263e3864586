"""The launch shapes that small env sets take (several warps per 32 envs in the step kernel,
8 envs per warp in the SIMT rollout, one to three 128-env tiles per block in the tensor-core
rollout) against the general shapes: the same arithmetic per env, so equal bit for bit."""
import numpy as np
import pytest
import torch

from helpers import cpu, lib_config
from test_gpu_env import _actor

pytestmark = pytest.mark.gpu

KEYS = ("state", "hist", "params", "dist", "ep_index", "ep_step", "ep_ret", "n_done", "records", "side")


def _bits(info, n, keys=KEYS):
    return [cpu(info[k])[..., :n].copy().view(np.uint32) for k in keys if k in info]


@pytest.mark.parametrize("n,n_hist,layout", [(1, 16, 0), (32, 16, 1), (33, 1, 3), (97, 0, 2), (64, 5, 0), (31, 0, 1)])
def test_step_writes_what_observe_reads(gpu, n, n_hist, layout):
    """The observations a step returns are those qsim_observe forms from the state it left,
    and the action history is the previous one shifted (zero after an episode end)."""
    q = gpu
    d, cfg, veh = lib_config(q, "c2", n_envs=n, capacity=8, critic_layout=layout, n_hist=n_hist, episode_len=4,
                             sig_p=0.01, sig_R=0.02, sig_v=0.03, sig_w=0.04, dist_f=0.01, dist_tau=1e-4)
    h = q.qsim_create(cfg, veh)
    try:
        info = q.qsim_info_get(h)
        ld, nh4 = info["ld"], 4 * n_hist
        buf = [torch.full((rows, ld), 7.0, device="cuda") for rows in
               (info["obs_dim"], info["critic_obs_dim"], info["obs_dim"], info["critic_obs_dim"])]
        for step in range(6):
            old = cpu(info["hist"]).copy()
            a = torch.rand(4, ld, device="cuda", generator=torch.Generator("cuda").manual_seed(step)) * 2.4 - 1.2
            q.qsim_step(h, a, buf[0], buf[1])
            q.qsim_observe(h, buf[2], buf[3])
            torch.cuda.synchronize()
            for x, y in ((0, 2), (1, 3)):
                assert np.array_equal(cpu(buf[x])[:, :n].view(np.uint32), cpu(buf[y])[:, :n].view(np.uint32))
            want = old.copy()
            want[4:nh4] = old[:max(nh4 - 4, 0)]
            if nh4:
                want[:4] = np.clip(cpu(a), -1, 1)
            ended = cpu(info["ep_step"])[:n] == 0
            want[:, :n][:, ended] = 0.0
            assert np.array_equal(cpu(info["hist"])[:, :n], want[:, :n])
        assert (cpu(info["n_done"])[:n] > 0).all()
    finally:
        q.qsim_destroy(h)


@pytest.mark.parametrize("hidden,n,n_hist,noise", [(32, 1, 16, 0.01), (32, 1000, 16, 0.0), (64, 33, 3, 0.01),
                                                   (64, 2500, 16, 0.01), (128, 40, 0, 0.01), (128, 1300, 16, 0.01)])
def test_few_envs_rollout_equals_32_per_warp(gpu, hidden, n, n_hist, noise):
    """An untuned handle of few envs runs 8 envs per warp; a handle with its warps per block
    pinned runs 32."""
    q = gpu
    outs = []
    for pinned in (0, 2):
        d, cfg, veh = lib_config(q, "c2", n_envs=n, capacity=30, learning_starts=2, n_hist=n_hist, episode_len=11,
                                 sig_p=noise, sig_v=noise, dist_f=0.01)
        h = q.qsim_create(cfg, veh)
        try:
            A = torch.tensor(_actor(d, hidden), device="cuda")
            q.qsim_rollout_engine(h, 1)
            if pinned:
                q.qsim_rollout_tune(h, pinned)
            q.qsim_rollout(h, A, hidden, 17, 0.1)
            q.qsim_rollout(h, A, hidden, 9, 0.0)
            torch.cuda.synchronize()
            outs.append(_bits(q.qsim_info_get(h), n))
        finally:
            q.qsim_destroy(h)
    for x, y in zip(*outs):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n", [1, 129, 152 * 128 + 1, 2 * 152 * 128 + 1])
def test_tensor_core_tiles_per_block_agree(gpu, n):
    """One, two or three tiles per block (chosen by the env count) against two partitions,
    which always run three."""
    q = gpu
    outs = []
    for parts in (0, 2):
        d, cfg, veh = lib_config(q, "c2", n_envs=n, capacity=12, learning_starts=1, episode_len=9, sig_p=0.01)
        h = q.qsim_create(cfg, veh)
        try:
            A = torch.tensor(_actor(d, 64), device="cuda")
            q.qsim_rollout_engine(h, 2)
            q.qsim_rollout_schedule(h, parts, 0)
            q.qsim_rollout(h, A, 64, 12, 0.1)
            q.qsim_sync(h)
            outs.append(_bits(q.qsim_info_get(h), n))
        finally:
            q.qsim_destroy(h)
    for x, y in zip(*outs):
        assert np.array_equal(x, y)
