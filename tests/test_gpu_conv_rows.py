"""The convolutions that march down grid rows, a kernel per layer: each against an fp64 convolution of the layer before it."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


def check(pol, layer, x, n, stride):
    """x: the layer's input.  Half a unit in the last place of fp16, and tensor-core sums cut off at 2^-22 of the terms, one per
    16 products and a few more."""
    w = torch.from_numpy(pol.params[f"conv{layer}_w"]).cuda().to(torch.bfloat16).double()
    b = torch.from_numpy(pol.params[f"conv{layer}_b"]).cuda().to(torch.bfloat16).double()
    got = torch.from_numpy(pol.activation(layer, n)).cuda().double()
    for at in range(0, n, 500):
        xs = torch.from_numpy(x[at:at + 500]).cuda().double()
        ref = torch.relu(torch.nn.functional.conv2d(xs, w, b, stride=stride))
        mag = torch.nn.functional.conv2d(xs, w.abs(), b.abs(), stride=stride)
        bound = 2.0 ** -11 * ref + (w[0].numel() / 16 + 8) * 2.0 ** -22 * mag + 2.0 ** -25
        assert bool((torch.abs(got[at:at + 500] - ref) <= bound).all()), (layer, at)


@pytest.mark.parametrize("C,H,W,sizes", [
    (8, 84, 84, (1, 12, 13, 14, 15, 128, 301)),     # 10 and 9 columns an environment: tiles of 128 end inside, at and past one
    (16, 72, 96, (1, 10, 32, 33, 150, 2500)),       # 12 and 10 columns; 2500: more output rows per block than accumulators
    (16, 36, 252, (1, 2, 5, 40)),                      # the widest frames: 31 and 30 columns
    (8, 160, 44, (2, 77)),                          # 20 grid rows: one tile is longer than the ring of accumulators
    (16, 52, 64, (3, 31, 62)),                      # 16 columns: a tile of 124 new ones is not a whole number of environments
    (4, 84, 84, (889, 1500, 3600))])                # 3600: the first layer's pipes share tiles
def test_layers(C, H, W, sizes):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W)
    pol = Policy(cfg, max_batch=max(sizes) + 3)
    try:
        for n in sizes:
            obs = wl.make_obs(cfg, n)
            out = pol.step(obs, np.arange(n, dtype=np.int32), 3, 17)
            assert np.isfinite(out["logits"]).all()
            check(pol, 1, obs / 255.0, n, 4)
            check(pol, 2, pol.activation(1, n), n, 2)
            check(pol, 3, pol.activation(2, n), n, 1)
    finally:
        pol.close()
