"""Training calls captured in a CUDA graph: their run descriptors are the graph's, whatever the
host memory they were made in holds when it is replayed."""
import numpy as np
import pytest
import torch

from helpers import cpu
from test_gpu_learner import NETS, make_run

pytestmark = pytest.mark.gpu


def _bits(q, runs):
    torch.cuda.synchronize()
    return [cpu(q.ac_info_get(a)[k]).view(np.uint32).copy() for a in runs for k in NETS]


@pytest.mark.parametrize("what", ["train", "update", "static"])
def test_captured_call_replays_its_own_descriptors(gpu, what):
    q = gpu

    def call(runs, envs):
        if what == "train":
            q.ac_train(runs, envs, 2)
        elif what == "update":
            q.ac_update(runs[0], envs[0], 2)
        else:
            q.ac_update_static(runs[0], envs[0], 2)

    sets = []
    try:
        for _ in range(2):
            made = [make_run(q, hidden=32, batch=32, cluster=1, seed=s) for s in range(3)]
            sets.append(([m[2] for m in made], [m[1] for m in made]))
        for runs, envs in sets:  # (the learner's own workspace is allocated before the capture)
            q.ac_update(runs[0], envs[0], 1)
        for _, envs in sets:  # a changed descriptor, so that a captured update uploads it
            q.qsim_step(envs[0], torch.zeros(4, q.qsim_info_get(envs[0])["ld"], device="cuda"))
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            call(*sets[0])
        # the memory that held the descriptors is used for something else
        junk = [np.full(1 << k, 0xA5, np.uint8) for k in range(6, 16) for _ in range(8)]
        g.replay()
        call(*sets[1])
        for got, want in zip(_bits(q, sets[0][0]), _bits(q, sets[1][0])):
            assert np.array_equal(got, want)
        del junk
    finally:
        for runs, envs in sets:
            for a, h in zip(runs, envs):
                q.ac_destroy(a)
                q.qsim_destroy(h)
