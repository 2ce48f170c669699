"""The gradient's tensor-core sums against 64 bits, given the ReLU decisions of the run itself; and with infinite inputs."""
import dataclasses

import numpy as np
import pytest
import torch
import torch.nn.functional as F

import hts_workloads as wl
from gpu_util import Policy
from test_gpu_backward import gpu_gradient, make_batch

pytestmark = pytest.mark.gpu
# A chain of eight products sums is cut off eight times, each time by less than one last place (2^-23) of what it holds.
# fp32 roundings of the rest go either way.  One chain for a whole range of rows (190 sums of conv1 at n = 640) is at 2.5 times that.
CHAIN = 8 * 2.0 ** -23


def gradient64(params, obs, actions, adv, ret, cv, ce, masks, chunk=128):
    """Actor-critic objective's gradient by library operations in 64 bits; masks: which hidden units pass."""
    w = {k: torch.from_numpy(np.asarray(v, np.float32)).cuda().double().requires_grad_() for k, v in params.items()}
    n, total = len(obs), {k: torch.zeros_like(v) for k, v in w.items()}
    f32 = lambda x: float(np.float32(x))
    for i in range(0, n, chunk):
        s = slice(i, min(n, i + chunk))
        x = torch.from_numpy(obs[s]).cuda().double() / 255
        for layer, stride in ((1, 4), (2, 2), (3, 1)):
            x = torch.where(masks[layer - 1][s], F.conv2d(x, w[f"conv{layer}_w"], w[f"conv{layer}_b"], stride), 0.0)
        h = torch.where(masks[3][s], F.linear(x.flatten(1), w["fc_w"], w["fc_b"]), 0.0)
        logp = F.linear(h, w["pi_w"], w["pi_b"]).log_softmax(1)
        v = F.linear(h, w["v_w"], w["v_b"])[:, 0]
        a = torch.from_numpy(np.asarray(actions[s], np.int64)).cuda()
        term = logp.gather(1, a[:, None])[:, 0] * torch.from_numpy(adv[s]).cuda().double()
        term = term - f32(cv) * (torch.from_numpy(ret[s]).cuda().double() - v) ** 2 - f32(ce) * (logp.exp() * logp).sum(1)
        for k, g in zip(w, torch.autograd.grad(term.sum() / n, list(w.values()))):
            total[k] += g
    return {k: v.cpu().numpy() for k, v in total.items()}


# stages per range of rows: one or two, three or four, and as many as a learner's largest batches have
@pytest.mark.parametrize("C,H,W,n", [(4, 84, 84, 80), (4, 84, 84, 150), (8, 84, 84, 640), (16, 72, 96, 61)])
def test_error_stays_within_one_chain(C, H, W, n):
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W)
    pol = Policy(cfg, max_batch=n)
    try:
        obs, actions, adv, ret = make_batch(cfg, n, n)
        got = gpu_gradient(pol, obs, actions, adv, ret, None, 0.5, 0.01, 0.0)
        masks = [torch.from_numpy(pol.activation(layer, n) > 0).cuda() for layer in (1, 2, 3, 4)]
        ref = gradient64(pol.params, obs, actions, adv, ret, 0.5, 0.01, masks)
        for k in ("conv1_w", "conv1_b", "conv2_w", "conv2_b", "conv3_w", "conv3_b", "fc_w", "fc_b"):
            e = np.linalg.norm(got[k] - ref[k]) / np.linalg.norm(ref[k])
            assert e <= CHAIN, (k, e, CHAIN)
    finally:
        pol.close()


@pytest.mark.parametrize("positive", [True, False])
def test_an_infinite_return_gives_infinities_where_fp32_sums_do(positive):
    """With every weight and pixel positive no infinities cancel and none meets a zero, so they reach all hidden layers'
    gradients as infinities; with weights of both signs some entries are NaN, some infinite, some finite."""
    n = 70
    cfg = wl.CONFIGS[1]
    params = wl.make_weights(cfg)
    if positive:
        params = {k: v if k.startswith("pi") else np.abs(v) for k, v in params.items()}
    pol = Policy(cfg, params=params, max_batch=n)
    try:
        obs, actions, adv, ret = make_batch(cfg, n, 5)
        obs = np.maximum(obs, 1)
        ret[66] = np.inf
        got = gpu_gradient(pol, obs, actions, adv, ret, None, 0.5, 0.01, 0.0)
        masks = [torch.from_numpy(pol.activation(layer, n) > 0).cuda() for layer in (1, 2, 3, 4)]
        ref = gradient64(pol.params, obs, actions, adv, ret, 0.5, 0.01, masks)
        kind = lambda x: np.where(np.isnan(x), 2, np.where(np.isinf(x), np.sign(x), 0))
        for k in ref:
            assert np.array_equal(kind(got[k]), kind(ref[k])), k
        if positive:
            assert all(np.all(got[f"{k}_{p}"] == np.inf) for k in ("conv1", "conv2", "conv3", "fc") for p in "wb")
        else:
            assert set(np.unique(kind(got["fc_w"]))) == {-1, 0, 1, 2}
    finally:
        pol.close()


# the passes that share a launch: more data-gradient tiles than blocks of them, row counts on both sides of a tile, one row
@pytest.mark.parametrize("C,H,W,n", [(4, 84, 84, 1), (4, 84, 84, 128), (4, 84, 84, 129), (4, 84, 84, 300), (16, 72, 96, 133), (4, 36, 44, 500)])
def test_passes_that_share_a_launch(C, H, W, n):
    test_error_stays_within_one_chain(C, H, W, n)
