"""fp32 layers in tiles: where rows leave strips half empty or are too wide for them, and dense layers of few features."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


def layers_us(H, W, n):
    """Device time of each layer of a step of n frames, the least of five rounds."""
    cfg = dataclasses.replace(wl.CONFIGS[1], H=H, W=W)
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = torch.zeros(n, cfg.C, H, W, dtype=torch.uint8, device="cuda"), torch.arange(n, dtype=torch.int32, device="cuda")
        out = [torch.empty(n, dtype=torch.int32, device="cuda")] + [torch.empty(n, device="cuda") for _ in range(3)]
        best = {}
        for _ in range(5):
            hts.hts_policy_profile(pol.ctx, True)
            for _ in range(10):
                hts.hts_policy_step(pol.ctx, obs, ids, None, 3, 17, n, *out, None)
            torch.cuda.synchronize()
            for k in range(5):
                ms, count = hts.hts_policy_profile_read(pol.ctx, k)
                name = hts.hts_policy_kernel_name(k)
                best[name] = min(best.get(name, 1e9), ms / count * 1e3)
            hts.hts_policy_profile(pol.ctx, False)
        return best
    finally:
        pol.close()


def check_bits(C, H, W, n):
    """The first and the last rows of a batch are the same bits as in a batch of their own, whose layers run in other forms."""
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W)
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        whole = pol.step(obs, ids, 3, 17)
        for at in (0, n - 8):
            few = pol.step(obs[at:at + 8], ids[at:at + 8], 3, 17)
            for k in whole:
                assert np.array_equal(whole[k][at:at + 8].view(np.int32), few[k].view(np.int32)), (at, k)
    finally:
        pol.close()


# a dense layer of 64 features: fewer columns than a box; more than five blocks of 16 rows per SM
@pytest.mark.parametrize("n", [81, 400, 2047])
def test_a_dense_layer_of_few_features(n):
    check_bits(4, 36, 36, n)


def test_a_quarter_of_the_features_takes_no_longer():
    assert layers_us(36, 36, 2048)["fc"] <= 1.1 * layers_us(44, 44, 2048)["fc"]


# the second layer's rows of 5 pixels in strips of 9, of 12, 14 and 16 in strips of 10, the third's of 3 in 4 and of 12 in 8; rows too wide; ragged ends
@pytest.mark.parametrize("C,H,W,n", [(4, 52, 52, 2047), (1, 112, 112, 515), (4, 128, 128, 512), (1, 144, 144, 509), (4, 48, 1024, 200),
                                     (4, 36, 36, 1183), (4, 36, 36, 1185), (1, 84, 36, 255)])      # the third's of one pixel: strips, tiles
def test_layers_whose_strips_are_half_empty_or_do_not_fit(C, H, W, n):
    check_bits(C, H, W, n)


def test_rows_too_wide_for_strips_take_no_longer_for_their_outputs():
    """504 outputs of each channel a frame in rows of 126 pixels, 372 in rows of 62."""
    wide, fits = layers_us(48, 1024, 200)["conv2"], layers_us(64, 512, 256)["conv2"]
    assert wide / (200 * 504) <= 1.25 * fits / (256 * 372)
