"""The heads in their forms (few rows per SM, several rows per warp, one warp per row): a row's outputs do not show which."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc
from gpu_util import Policy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("A", [2, 7, 8, 18, 31, 32, 33, 63, 64])       # outputs A + 1: eight to a pass, actions 32 to a lane
def test_forms(A):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=4, H=36, W=44, A=A)
    n = 4800                                             # four rows a warp
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        full = pol.step(obs, ids, 3, 17)
        for m in (1, 3, 149, 592, 593, 1184, 1185, 4701):        # the last: two rows a warp
            rows = np.arange(n - m, n)
            part = pol.step(obs[rows], ids[rows], 3, 17)
            for k in full:
                assert np.array_equal(part[k].view(np.int32), full[k][rows].view(np.int32)), (m, k)
        for e in (0, 1, 2, 3, n - 1):                    # fp32 rounding of the distribution, given the logits
            lp, ent = orc.log_softmax(full["logits"][e].astype(np.float64))
            assert abs(full["logp"][e] - lp[full["actions"][e]]) <= 2e-5 * max(1.0, abs(lp[full["actions"][e]]))
            assert abs(full["entropy"][e] - ent) <= 2e-5 * max(1.0, ent)
    finally:
        pol.close()


def test_given_actions():
    cfg = dataclasses.replace(wl.CONFIGS[1], C=4, H=36, W=44)
    n = 5000
    pol = Policy(cfg, max_batch=n)
    try:
        obs = torch.from_numpy(wl.make_obs(cfg, n)).cuda()
        act = (torch.arange(n, device="cuda") % cfg.A).to(torch.int32)

        def evaluate(rows):
            out = [torch.empty(rows.numel(), device="cuda") for _ in range(3)]
            hts.hts_policy_evaluate(pol.ctx, obs[rows].contiguous(), act[rows].contiguous(), rows.numel(), *out)
            return torch.stack(out)

        full = evaluate(torch.arange(n, device="cuda"))
        for m in (1, 592, 593, 1184, 1185, 1777, 4737):
            assert torch.equal(evaluate(torch.arange(n - m, n, device="cuda")), full[:, n - m:]), m
    finally:
        pol.close()
