"""The reverse sweep refuses a workspace smaller than its descriptor's before anything is launched
(runs without a GPU)."""
import pytest
import torch

import paper_2311_13081_gb300 as q
from paper_2311_13081_gb300 import diff


@pytest.mark.parametrize("change", [dict(H=64), dict(ckpt=23), dict(n_hist=16)])
def test_workspace_of_another_descriptor_is_refused(change):
    base = dict(n=64, ld=64, H=23, ckpt=10, mode=1, weights=(1.0, 1.0, 1.0, 1.0), n_hist=4, hidden=32)
    ws = torch.empty(q.qsim_vjp_workspace(diff.make_desc(**base)) // 4)
    desc = diff.make_desc(**{**base, **change})
    assert q.qsim_vjp_workspace(desc) > 4 * ws.numel()
    with pytest.raises(ValueError, match="workspace of"):
        q.qsim_rollout_vjp_reverse(desc, q.QsimParams(), None, None, None, None, None, None, None, None, ws)
