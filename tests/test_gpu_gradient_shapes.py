"""The gradient's tensor-core tiles at batch and frame sizes where they change: remainders of a tile, channels that are
padded, grids so wide that every filter tap loads its own rows, a batch smaller than the previous one."""
import dataclasses

import numpy as np
import pytest

import hts_workloads as wl
from gpu_util import Policy
from test_gpu_backward import check, gpu_gradient, make_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W,A,n", [(1, 36, 36, 2, 1), (3, 44, 60, 7, 9), (4, 84, 84, 64, 22), (20, 40, 48, 5, 6),
                                       (4, 36, 256, 6, 3), (4, 36, 532, 6, 3), (6, 40, 1040, 3, 2)])
def test_frame_shapes(C, H, W, A, n):
    cfg = dataclasses.replace(wl.CONFIGS[1], C=C, H=H, W=W, A=A)
    pol = Policy(cfg, max_batch=n + 3)
    try:
        obs, actions, adv, ret = make_batch(cfg, n, H + W + n)
        check(pol, obs, actions, adv, ret, None, 0.5, 0.01, 0.0)
    finally:
        pol.close()


def test_rows_of_an_earlier_batch_do_not_leak_in():
    cfg = wl.CONFIGS[1]
    pol, fresh = Policy(cfg, max_batch=70), Policy(cfg, max_batch=70)
    try:
        obs, actions, adv, ret = make_batch(cfg, 70, 3)
        gpu_gradient(pol, obs, actions, adv, ret, None, 0.5, 0.01, 0.0)
        for n in (1, 13, 65):
            a = gpu_gradient(pol, obs[:n], actions[:n], adv[:n], ret[:n], None, 0.5, 0.01, 0.0)
            b = gpu_gradient(fresh, obs[:n], actions[:n], adv[:n], ret[:n], None, 0.5, 0.01, 0.0)
            for k in a:
                assert np.array_equal(a[k].view(np.int32), b[k].view(np.int32)), (n, k)
    finally:
        pol.close(); fresh.close()
