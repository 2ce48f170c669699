"""Weight gradients of the heads for few samples: no further from 64 bits than the sums of a launch of their own, which larger batches take."""
import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy
from test_gpu_backward import gpu_gradient, make_batch

pytestmark = pytest.mark.gpu
f32, f64 = np.float32, np.float64


def ranges_of_sixteen(d, h):
    """Chains of every fourth sample of a range, products not rounded before they are added; the ranges in quarters."""
    parts = []
    for i in range(0, len(d), 16):
        chain = np.zeros((4, h.shape[1]), f32)
        for k in range(i, min(i + 16, len(d))):
            chain[k % 4] = (d[k].astype(f64) * h[k].astype(f64) + chain[k % 4]).astype(f32)
        parts.append((chain[0] + chain[1]) + (chain[2] + chain[3]))
    q = [sum(parts[len(parts) * k // 4:len(parts) * (k + 1) // 4], np.zeros(h.shape[1], f32)) for k in range(4)]
    return (q[0] + q[1]) + (q[2] + q[3])


# one sample, less than a range, whole ranges, ragged ones, as many as are summed without a launch of their own
@pytest.mark.parametrize("n", [1, 7, 16, 20, 41, 64, 79, 80])
def test_value_weights_of_few_samples(n):
    """With a value coefficient of 1/2 a sample's factor is (return - value) / n, known to the bit."""
    cfg = wl.CONFIGS[1]
    pol = Policy(cfg, max_batch=n)
    try:
        obs, actions, adv, ret = make_batch(cfg, n, n)
        got = gpu_gradient(pol, obs, actions, np.zeros_like(adv), ret, None, 0.5, 0.0, 0.0)
        h = pol.activation(4, n)
        out = [torch.empty(n, device="cuda") for _ in range(3)]
        hts.hts_policy_evaluate(pol.ctx, torch.from_numpy(obs).cuda(), torch.from_numpy(actions.astype(np.int32)).cuda(), n, *out)
        d = ((ret - out[1].cpu().numpy()) * (f32(1) / f32(n))).astype(f32)
    finally:
        pol.close()
    ref = (d.astype(f64)[:, None] * h).sum(0)
    error = lambda x: np.linalg.norm(x.reshape(-1) - ref)
    assert error(got["v_w"]) <= 1.001 * error(ranges_of_sixteen(d, h)), (error(got["v_w"]), error(ranges_of_sixteen(d, h)))
    # the biases' chains are no longer
    assert abs(got["v_b"].item() - d.astype(f64).sum()) <= 22 * 2.0 ** -24 * np.abs(d).sum()
