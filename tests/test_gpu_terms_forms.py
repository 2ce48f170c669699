"""Standardised sample means on both sides of the counts where the kernel of sums changes its form: two blocks of 2048 transitions
per SM, three, and as many blocks as there are (from there on a thread has more than two groups)."""
import pytest
import torch

import paper_2012_09849_b200 as hts

pytestmark = pytest.mark.gpu


def check(count, aligned):
    g = torch.Generator(device="cuda").manual_seed(count)
    x = [torch.randn(count + 1, device="cuda", generator=g) for _ in range(6)]
    x[1] = x[0] + 0.2 * x[1]
    x = [a[:count] if aligned else a[1:] for a in x]
    out = torch.empty(2, 4, device="cuda")
    for k in range(2):                                   # the second call follows the first without a pause
        hts.hts_ppo_terms(*x, count, 0.2, True, out[k])
    ln, lo, v, h, a, r = [y.double() for y in x]
    a = (a - a.mean()) / (a.std(unbiased=False) + 1e-8)
    rho, clip = (ln - lo).exp(), torch.tensor(0.2, dtype=torch.float32).double().item()
    ref = [torch.minimum(rho * a, rho.clamp(1 - clip, 1 + clip) * a).mean(), ((r - v) ** 2).mean(), h.mean()]
    scale = [(rho * a).abs().mean(), ref[1], h.abs().mean()]
    assert torch.equal(out[0], out[1])
    for k in range(3):                                   # the ratio is an fp32 exponential of an fp32 difference: 2^-21 of a term
        assert abs(out[0, k].item() - ref[k].item()) <= 2.0 ** -20 * scale[k].item(), k
    # of the ratios, that exponential moves about one in a million across the edge of the clip range
    assert abs(out[0, 3].item() - ((rho - 1).abs() > clip).double().mean().item()) <= 2e-6 + 2.0 / count


@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("blocks_per_sm,blocks", [(2, 0), (3, 0), (0, 2048)])
@pytest.mark.parametrize("more", [-3, 0, 1, 2053])
def test_against_64_bits(blocks_per_sm, blocks, more, aligned):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    check((blocks or blocks_per_sm * sms) * 2048 + more, aligned)


# one block, more blocks, ragged ends and blocks without a transition, as many as the blocks' shared memory holds, and one more
@pytest.mark.parametrize("aligned", [True, False])
@pytest.mark.parametrize("count", [1, 3, 4, 7, 512, 513, 2047, 2049, 8191, 8193, 70001, 147453, 147456, 147457])
def test_few_transitions_against_64_bits(count, aligned):
    check(count, aligned)
