"""The two scans' forms for tall problems: the chain of chunk maps walked by the first warp, blocks alone on their SM."""
import numpy as np
import pytest
import torch

import paper_2012_09849_b200 as hts
from oracle import hts_oracle as orc

pytestmark = pytest.mark.gpu


def problem(T, N, seed):
    g = np.random.default_rng(seed)
    return [(g.random((T, N)) < 0.1).astype(np.float32), g.standard_normal((T, N)).astype(np.float32), (g.random((T, N)) < 0.02).astype(np.uint8),
            g.standard_normal(N).astype(np.float32), (0.3 * g.standard_normal((T, N))).astype(np.float32)]


def scans(r, v, d, b, lr):
    T, N = r.shape
    dev = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (r, v, d, b, lr)]
    out = [torch.full((T, N), float("nan"), device="cuda") for _ in range(4)]
    hts.hts_gae(*dev[:4], 0.99, 0.95, T, N, *out[:2])
    hts.hts_vtrace(dev[4], *dev[:4], 0.99, 0.95, 1.0, 1.0, T, N, *out[2:])
    torch.cuda.synchronize()
    return [x.cpu().numpy() for x in out]


# chunks of eight rows: 31, 32 and 33 of them, the last ones ragged, and more than a block's warps take in one step
@pytest.mark.parametrize("T", [241, 248, 249, 256, 257, 511, 513, 700, 1100])
@pytest.mark.parametrize("N", [1, 8, 37, 1200])
def test_tall_scans_have_the_bits_of_wide_ones(T, N):
    wide = problem(T, 5000, T)                           # several blocks per SM, few chunks per step
    narrow = [x[..., :N] for x in wide]
    got = scans(*narrow)
    for a, b in zip(got, scans(*wide)):
        assert np.array_equal(a.view(np.int32), np.ascontiguousarray(b[:, :N]).view(np.int32))
    r, v, d, b, _ = (np.ascontiguousarray(x[..., :8]) for x in wide)
    adv, ret = orc.gae(r, v, d, b, np.float32(0.99), np.float32(0.95))
    k = min(N, 8)
    for a, ref in ((got[0], adv), (got[1], ret)):        # fp32 recurrences of length T that forget at 0.94 a step: 17 steps' roundings
        assert np.abs(a[:, :k] - ref[:, :k]).max() <= 1e-5 * max(1.0, np.abs(ref).max())
