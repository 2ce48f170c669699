"""Both scans on either side of each change of block shape: columns per block, chunks per step, rows that end inside a
chunk or a step; and the one-pass advantage statistics where the mean dwarfs the spread."""
import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc
from gpu_util import gpu_gae, rel_err

pytestmark = pytest.mark.gpu
SHAPES = [(31, 40), (32, 2368), (513, 33), (1030, 9), (20, 4736), (137, 4737), (65, 18912), (66, 18945), (9, 37889), (56, 75776), (60, 75772)]


@pytest.mark.parametrize("T,N", SHAPES)
def test_advantages(T, N):
    r, v, d, b = wl.make_rollout(wl.CONFIGS[4], T=T, N=N, sub=T + N)
    adv, ret = gpu_gae(r, v, d, b, 0.99, 0.95)
    a_ref, r_ref = orc.gae(r, v, d, b, float(np.float32(0.99)), float(np.float32(0.95)))
    assert rel_err(adv, a_ref) <= 1e-5 and rel_err(ret, r_ref) <= 1e-5


@pytest.mark.parametrize("T,N", SHAPES)
def test_vtrace(T, N):
    r, v, d, b = wl.make_rollout(wl.CONFIGS[4], T=T, N=N, sub=T + N)
    lr = (0.3 * np.random.default_rng(T * N).standard_normal((T, N))).astype(np.float32)
    g = [torch.from_numpy(x).cuda() for x in (lr, r, v, d, b)]
    vs, pg = torch.empty(T, N, device="cuda"), torch.empty(T, N, device="cuda")
    hts.hts_vtrace(*g, 0.99, 0.95, 1.0, 0.9, T, N, vs, pg)
    f = lambda x: float(np.float32(x))
    vs_ref, pg_ref = orc.vtrace(lr, r, v, d, b, f(0.99), f(0.95), 1.0, f(0.9))
    assert rel_err(vs.cpu().numpy(), vs_ref) <= 1e-5 and rel_err(pg.cpu().numpy(), pg_ref) <= 1e-5


@pytest.mark.parametrize("mean,count", [(0.0, 1), (1e4, 2049), (-3e5, 100003)])
def test_standardised_advantages_far_from_zero(mean, count):
    g = np.random.default_rng(count)
    x = [g.standard_normal(count).astype(np.float32) for _ in range(6)]
    x[4] = (x[4] + np.float32(mean)).astype(np.float32)
    out = torch.empty(4, device="cuda")
    hts.hts_ppo_terms(*[torch.from_numpy(a).cuda() for a in x], count, 0.2, True, out)
    a = x[4].astype(np.float64)
    a = (a - a.mean()) / (a.std() + 1e-8)
    rho = np.exp((x[0] - x[1]).astype(np.float64))
    clip = float(np.float32(0.2))
    ref = np.minimum(rho * a, np.clip(rho, 1 - clip, 1 + clip) * a).mean()
    assert abs(float(out[0]) - ref) <= 1e-5 * max(1.0, abs(ref))
