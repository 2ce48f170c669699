"""The fp32 actor step's tiles: batch sizes on both sides of every tile and of every change of tile shape."""
import dataclasses

import numpy as np
import pytest

import hts_workloads as wl
from oracle import hts_oracle as orc
from gpu_util import Policy, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W,sizes", [
    (4, 84, 84, (1, 15, 16, 17, 32, 33, 72, 80, 81, 128, 129, 200, 384, 700)),     # every tile of the convolutions and of the dense layer
    (3, 36, 44, (1, 20, 33, 400)),                       # channels not a multiple of four, a dense layer of 256 features
    (16, 72, 96, (2, 130))])
def test_rows_do_not_depend_on_the_tile(C, H, W, sizes):
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W)
    n = max(sizes)
    pol = Policy(cfg, max_batch=n)
    try:
        obs = wl.make_obs(cfg, n)
        ids = np.arange(n, dtype=np.int32)
        full = pol.step(obs, ids, 3, 17)
        for m in sizes:
            rows = np.arange(n - m, n)                   # the batch's last rows: other positions in other tiles
            part = pol.step(obs[rows], ids[rows], 3, 17)
            for k in full:
                assert np.array_equal(part[k].view(np.int32), full[k][rows].view(np.int32)), (m, k)
        rows = np.unique(np.array([0, n // 2, n - 1]))
        ref = orc.policy_step(orc.Weights(pol.params), obs[rows], ids[rows], 3, 17)
        assert rel_err(full["logits"][rows], ref["logits"]) <= 1e-4
    finally:
        pol.close()
