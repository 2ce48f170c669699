"""Both scans where wide problems change from blocks of 32 columns to blocks of 128, and the standardised terms where a thread
has no, one, two or more groups of the loads that are under way before the advantage statistics."""
import numpy as np
import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc
from gpu_util import gpu_gae, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,N", [(63, 80000), (64, 80000), (64, 113660), (64, 113664), (64, 151548), (64, 151552)])
def test_scans(T, N):
    r, v, d, b = wl.make_rollout(wl.CONFIGS[4], T=T, N=N, sub=T + N)
    f = lambda x: float(np.float32(x))
    adv, ret = gpu_gae(r, v, d, b, 0.99, 0.95)
    a_ref, r_ref = orc.gae(r, v, d, b, f(0.99), f(0.95))
    assert rel_err(adv, a_ref) <= 1e-5 and rel_err(ret, r_ref) <= 1e-5
    lr = (0.3 * np.random.default_rng(T * N).standard_normal((T, N))).astype(np.float32)
    vs, pg = torch.empty(T, N, device="cuda"), torch.empty(T, N, device="cuda")
    hts.hts_vtrace(*[torch.from_numpy(x).cuda() for x in (lr, r, v, d, b)], 0.99, 0.95, 1.0, 0.9, T, N, vs, pg)
    vs_ref, pg_ref = orc.vtrace(lr, r, v, d, b, f(0.99), f(0.95), 1.0, f(0.9))
    assert rel_err(vs.cpu().numpy(), vs_ref) <= 1e-5 and rel_err(pg.cpu().numpy(), pg_ref) <= 1e-5


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("count", [1, 3, 5, 1023, 1028, 2047, 2053, 131071, 131076, 4194304 + 7, 9000001])
def test_standardised_terms(count, aligned):
    g = torch.Generator(device="cuda").manual_seed(count)
    x = [torch.randn(count + 1, device="cuda", generator=g) for _ in range(6)]
    x[1] = x[0] + 0.2 * x[1]
    x = [a[:count] if aligned else a[1:] for a in x]
    out = torch.empty(4, device="cuda")
    for _ in range(2):                                   # the second call follows the first without a pause
        hts.hts_ppo_terms(*x, count, 0.2, True, out)
    ln, lo, v, h, a, r = [y.double() for y in x]
    a = (a - a.mean()) / (a.std(unbiased=False) + 1e-8)
    rho, clip = torch.exp(ln - lo), float(np.float32(0.2))
    s = torch.minimum(rho * a, rho.clamp(1 - clip, 1 + clip) * a)
    # the ratio is an fp32 exponential of an fp32 difference (2 and 1/2 ulp, of arguments up to about 1): 2^-21 of a term
    ref = [s.mean(), ((r - v) ** 2).mean(), h.mean()]
    scale = [(rho * a).abs().mean(), ref[1], h.abs().mean()]
    for k in range(3):
        assert abs(float(out[k]) - float(ref[k])) <= 2.0 ** -20 * float(scale[k]) + 1e-12, k
    # ratios at the edge of the clip range may fall either way: the fp32 exponential moves about one in a million across it
    assert abs(float(out[3]) - float(((rho - 1).abs() > clip).double().mean())) <= 2e-6 + 2.0 / count * (count > 100000)
