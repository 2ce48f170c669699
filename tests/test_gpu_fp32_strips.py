"""fp32 convolutions in strips against the gathered tiles: the same chain of sums per output, so the same bits."""
import dataclasses

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc
from gpu_util import Policy, rel_err

pytestmark = pytest.mark.gpu


def outputs(cfg, n):
    return torch.empty(n, dtype=torch.int32, device="cuda"), [torch.empty(n, device="cuda") for _ in range(3)], torch.empty(n, cfg.A, device="cuda")


@pytest.mark.parametrize("C,H,W,n", [
    (4, 84, 84, 1), (4, 84, 84, 43), (4, 64, 96, 39), (16, 72, 96, 31),      # rows of 20 / 9 / 7 and of 23 / 10 / 8
    (3, 36, 44, 200), (1, 36, 36, 250), (8, 44, 52, 90), (5, 60, 60, 90),    # odd channels, strips wider than a row
    (2, 40, 128, 40), (4, 132, 44, 40),                                      # rows of several strips, frames of many rows
    (2, 36, 512, 9)])
def test_strips_have_the_bits_of_the_tiles(C, H, W, n):
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W)
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        strips = pol.step(obs, ids, 3, 17)
        d_obs, d_ids = torch.from_numpy(obs).cuda(), torch.from_numpy(ids).cuda()
        act, f, logits = outputs(cfg, n)
        hts.hts_policy_step_noalloc(C, H, W, cfg.A, pol.dev_w, d_obs, d_ids, None, 3, 17, n, act, *f, logits)     # weights in the caller's layout: tiles
        torch.cuda.synchronize()
        tiles = {"actions": act, "logp": f[0], "values": f[1], "entropy": f[2], "logits": logits}
        for k, v in tiles.items():
            assert np.array_equal(strips[k].view(np.int32), v.cpu().numpy().view(np.int32)), k
        ref = orc.policy_step(orc.Weights(pol.params), obs[:2], ids[:2], 3, 17)
        assert rel_err(strips["logits"][:2], ref["logits"]) <= 1e-4
        for layer in (1, 2):                                                   # rows lie apart in the workspace
            got = pol.activation(layer, n)
            assert np.all(np.isfinite(got)) and got.max() > 0
    finally:
        pol.close()


@pytest.mark.parametrize("n", [5, 300, 1100])
@pytest.mark.parametrize("offset", [1, 4])
def test_frames_at_any_address(n, offset):
    """Frames that bulk copies cannot take go through the tiles, the other layers through strips."""
    cfg = wl.CONFIGS[1]
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        want = pol.step(obs, ids, 3, 17)
        buf = torch.empty(obs.size + 16, dtype=torch.uint8, device="cuda")
        view = buf[offset:offset + obs.size].view(obs.shape)
        view.copy_(torch.from_numpy(obs))
        act, f, logits = outputs(cfg, n)
        hts.hts_policy_step(pol.ctx, view, torch.from_numpy(ids).cuda(), None, 3, 17, n, act, *f, logits)
        torch.cuda.synchronize()
        assert np.array_equal(logits.cpu().numpy().view(np.int32), want["logits"].view(np.int32))
        assert np.array_equal(act.cpu().numpy(), want["actions"])
    finally:
        pol.close()


@pytest.mark.parametrize("C,H,W,sizes", [(4, 84, 84, (30, 50, 100)), (16, 72, 96, (30, 50, 100)), (2, 40, 128, (40, 150))])
def test_strips_of_five_pixels(C, H, W, sizes):
    """Batches of which the first layer's blocks of four-pixel strips take one round more than those of five."""
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W)
    n = max(sizes)
    pol = Policy(cfg, max_batch=n)
    try:
        obs, ids = wl.make_obs(cfg, n), np.arange(n, dtype=np.int32)
        few = [pol.step(obs[i:i + 8], ids[i:i + 8], 3, 17) for i in (0, n - 8)]
        for m in sizes:
            part = pol.step(obs[n - m:], ids[n - m:], 3, 17)
            for k in part:
                assert np.array_equal(part[k][-8:].view(np.int32), few[1][k].view(np.int32)), (m, k)
                if m == n:
                    assert np.array_equal(part[k][:8].view(np.int32), few[0][k].view(np.int32)), (m, k)
    finally:
        pol.close()
