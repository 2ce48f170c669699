"""Small batches of four-channel frames take one kernel for all three convolutions, larger ones a kernel per layer; and the
first convolution cuts its output rows into ranges that depend on the batch.  Neither may show in any bit."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc
from gpu_util import Policy, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W,sizes", [
    (4, 84, 84, (1, 2, 147, 149, 297, 592, 888, 889)),   # environments per SM; 889 is the first batch of the other kernels
    (4, 64, 96, (1, 150, 300)),                          # odd-sized hidden grids: border positions nothing writes
    (4, 36, 44, (1, 75, 160)),                           # too small for the shared kernel: its shifted tiles reach too far
    (4, 60, 60, (1, 150, 444, 445)),                     # two conv1 tiles, grids that fill little of a tile
    (16, 72, 96, (1, 3, 30, 149, 600)),                  # 17 output rows: ranges that do not divide them
    (8, 84, 84, (1, 20, 333))])
def test_batch_size_does_not_show(C, H, W, sizes):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W)
    n = 1000
    pol = Policy(cfg, max_batch=n)
    try:
        obs = wl.make_obs(cfg, n)
        ids = np.arange(n, dtype=np.int32)
        full = pol.step(obs, ids, 3, 17)
        for m in sizes:
            rows = np.arange(n - m, n)
            part = pol.step(obs[rows], ids[rows], 3, 17)
            for k in full:
                assert np.array_equal(part[k].view(np.int32), full[k][rows].view(np.int32)), (m, k)
        m = sizes[0] + 1                                 # the hidden layers of a small batch, with the parity taps
        pol.step(obs[:m], ids[:m], 3, 17)
        taps = orc.policy_forward(orc.Weights(pol.params), obs[:m], taps=True)
        for layer, name in ((1, "conv1"), (2, "conv2"), (3, "conv3"), (4, "fc")):
            assert rel_err(pol.activation(layer, m), taps[name]) <= 2e-2, name
    finally:
        pol.close()


@pytest.mark.parametrize("H,W,per_sm", [(88, 36, 3), (60, 60, 3), (84, 84, 5), (36, 44, 0)])
def test_largest_shared_batch(H, W, per_sm):
    """One kernel for the convolutions up to a number of observations per SM: three launches a step, five above."""
    cfg = dataclasses.replace(wl.CONFIGS[2], C=4, H=H, W=W)
    line = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    pol = Policy(cfg, max_batch=line + 1)
    try:
        for n, launches in ((line, 3), (line + 1, 5)):
            if n:
                before = hts.hts_launch_count()
                pol.step(np.zeros((n, 4, H, W), np.uint8), np.arange(n, dtype=np.int32), 0, 1)
                assert hts.hts_launch_count() - before == launches, n
    finally:
        pol.close()
