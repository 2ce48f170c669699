"""The dense layer's forms (resident weights; pairs of SMs with one, several or all K ranges): each against an fp64 product of
the layer's own input, and none of them to be told from another by a bit of the outputs."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
from gpu_util import Policy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W,sizes", [
    # seven ranges of seven chunks: resident to 640 rows, one range a pair to 1280, then three, two and one pair a 256 x 128
    # tile, 256 x 256 tiles above 4608
    (4, 84, 84, (640, 641, 769, 1024, 1025, 1280, 1281, 1536, 1537, 2304, 2305, 4608, 4609)),
    (4, 36, 44, (1, 129, 600, 2600)),                    # two ranges of one chunk
    (8, 84, 60, (1, 300, 700))])                         # 28 chunks: seven ranges of four
def test_forms(C, H, W, sizes):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W)
    n = max(sizes) + 200
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        full = pol.step(obs, ids, 3, 17)
        w = torch.from_numpy(pol.params["fc_w"]).cuda().to(torch.bfloat16).double()
        b = torch.from_numpy(pol.params["fc_b"]).cuda().to(torch.bfloat16).double()
        for m in sizes:
            rows = np.arange(n - m, n)
            part = pol.step(obs[rows], ids[rows], 3, 17)
            for k in full:
                assert np.array_equal(part[k].view(np.int32), full[k][rows].view(np.int32)), (m, k)
            x = torch.from_numpy(pol.activation(3, m)).cuda().double().flatten(1)
            got = torch.from_numpy(pol.activation(4, m)).cuda().double()
            # fp32 sums in tensor memory and of the ranges, each cut off or rounded at 2^-22 of the terms so far
            bound = (x.shape[1] / 16 + 8) * 2.0 ** -22 * (x.abs() @ w.abs().T + b.abs())
            assert bool((torch.abs(got - torch.relu(x @ w.T + b)) <= bound).all()), m
    finally:
        pol.close()
