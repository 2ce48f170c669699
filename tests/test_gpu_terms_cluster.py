"""Standardised sample means by one cluster of blocks, where more than the count decides what it meets."""
import ctypes

import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


def inputs(count):
    g = torch.Generator(device="cuda").manual_seed(count)
    x = [torch.randn(count, device="cuda", generator=g) for _ in range(6)]
    x[1] = x[0] + 0.2 * x[1]
    return x


# one block, a few, and sixteen
@pytest.mark.parametrize("count", [300, 2047, 131071])
def test_the_same_bits_beside_actor_steps(count):
    n, x = 1024, inputs(count)
    alone, beside = torch.empty(4, device="cuda"), torch.empty(50, 4, device="cuda")
    hts.hts_ppo_terms(*x, count, 0.2, True, alone)
    pol = Policy(wl.CONFIGS[3], max_batch=n)
    try:
        obs, ids = torch.from_numpy(wl.make_obs(wl.CONFIGS[3], n)).cuda(), torch.arange(n, dtype=torch.int32, device="cuda")
        out = [torch.empty(n, dtype=torch.int32, device="cuda")] + [torch.empty(n, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        actor, learner = torch.cuda.Stream(), torch.cuda.Stream()
        for k in range(50):
            hts.hts_policy_step(pol.ctx, obs, ids, None, k, 1, n, *out, None, actor.cuda_stream)
            hts.hts_ppo_terms(*x, count, 0.2, True, beside[k], learner.cuda_stream)
        torch.cuda.synchronize()
        assert hts.hts_last_async_error(pol.ctx) == 0
    finally:
        pol.close()
    assert np.array_equal(beside.cpu().numpy().view(np.int32), np.tile(alone.cpu().numpy().view(np.int32), (50, 1)))


def selftest(x, count, lost, out):
    f = hts.lib().hts_ppo_terms_selftest
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_void_p] * 6 + [ctypes.c_int64, ctypes.c_float, ctypes.c_int32] + [ctypes.c_void_p] * 2
    assert f(*(a.data_ptr() for a in x), count, 0.2, lost, out.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0


def test_copies_that_never_land_are_read_where_they_are():
    """The wait for them runs out after a moment; the result is the same, to the bit."""
    for count in (3, 700, 9217, 131071):
        x, out = inputs(count), torch.zeros(2, 4, device="cuda")
        hts.hts_ppo_terms(*x, count, 0.2, True, out[0])
        selftest(x, count, 1, out[1])
        torch.cuda.synchronize()
        assert np.array_equal(out[0].cpu().numpy().view(np.int32), out[1].cpu().numpy().view(np.int32)), count


# where the device has no room for the cluster: one thread, one block, more blocks, ragged ends, the most that the cluster takes
@pytest.mark.parametrize("count", [1, 3, 4, 511, 2048, 2049, 70001, 147456])
def test_two_launches_instead(count):
    """Both forms add the same terms in 64 bits, so that they differ by the rounding of the result to 32."""
    x, out = inputs(count), torch.zeros(2, 4, device="cuda")
    hts.hts_ppo_terms(*x, count, 0.2, True, out[0])
    selftest(x, count, 0, out[1])
    a, b = out.double().cpu().numpy()
    rho = (x[0] - x[1]).double().exp()
    z = (x[4].double() - x[4].double().mean()) / (x[4].double().std(unbiased=False) + 1e-8)
    scale = np.array([(rho * z).abs().mean().item(), a[1], x[3].abs().mean().item(), 0.0])
    assert np.all(np.abs(a - b) <= 2.0 ** -23 * np.abs(a) + 2.0 ** -36 * scale), (a, b)
