"""The two scans where every block carries from super-chunk to super-chunk: few columns against so many that each thread walks the chunk maps."""
import numpy as np
import pytest
import torch

from oracle import hts_oracle as orc
from test_gpu_scan_chain import problem, scans

pytestmark = pytest.mark.gpu


# one super-chunk of the forms for few columns, a little more than one, several; 4 blocks of 32 columns per SM and more
@pytest.mark.parametrize("T", [249, 257, 513, 1100])
def test_few_columns_have_the_bits_of_many(T):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    wide = problem(T, 32 * 4 * sms + 32, T)
    want = scans(*wide)
    for N in (8, 37, 1200, 32 * sms - 5, 32 * sms):      # 8-column blocks, and 32-column blocks up to one per SM
        got = scans(*(x[..., :N] for x in wide))
        for a, b in zip(got, want):
            assert np.array_equal(a.view(np.int32), np.ascontiguousarray(b[:, :N]).view(np.int32)), N
    r, v, d, b, lr = (np.ascontiguousarray(x[..., :8]) for x in wide)
    f = np.float32
    ref = orc.gae(r, v, d, b, f(0.99), f(0.95)) + orc.vtrace(lr, r, v, d, b, f(0.99), f(0.95), f(1), f(1))
    # a step rounds five times and has an exponential of two ulps, 5.4e-7 of its terms; recurrences that forget at 0.94 a step
    # gather 17 steps; policy-gradient advantages have up to two such terms
    for a, x in zip(want, ref):
        assert np.abs(a[:, :8] - x).max() <= 2e-5 * max(1.0, np.abs(x).max())
