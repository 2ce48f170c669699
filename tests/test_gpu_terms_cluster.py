"""Standardised sample means by one cluster of blocks, where more than the count decides what it meets."""
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


def test_copies_that_never_land_are_read_where_they_are():
    """The wait for them runs out after a moment; the result is the same, to the bit."""
    import ctypes
    selftest = hts.lib().hts_ppo_terms_selftest
    selftest.restype, selftest.argtypes = ctypes.c_int, [ctypes.c_void_p] * 6 + [ctypes.c_int64, ctypes.c_float] + [ctypes.c_void_p] * 2
    for count in (3, 700, 9217, 131071):
        x, out = inputs(count), torch.zeros(2, 4, device="cuda")
        hts.hts_ppo_terms(*x, count, 0.2, True, out[0])
        assert selftest(*(a.data_ptr() for a in x), count, 0.2, out[1].data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
        torch.cuda.synchronize()
        assert np.array_equal(out[0].cpu().numpy().view(np.int32), out[1].cpu().numpy().view(np.int32)), count
