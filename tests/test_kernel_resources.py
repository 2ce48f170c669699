"""Registers and spills of kernels whose launch counts on a number of blocks per SM (what the compiler reports; no GPU)."""
import os
import re
import subprocess

import pytest

from paper_2012_09849_b200 import build as hb

REGISTERS_PER_SM, THREADS = 65536, 256


def compiled(source):
    """{mangled entry: (registers, spilled bytes)} of one source file."""
    cmd = [os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3",
           "-std=c++17", "-I", os.path.join(hb.ROOT, "include"), "-Xptxas", "-v", "-cubin", "-o", os.devnull,
           os.path.join(hb.PKG, "csrc", source)]
    text = subprocess.run(cmd, check=True, capture_output=True, text=True).stderr
    out = {}
    for part in text.split("Compiling entry function '")[1:]:
        used = int(re.search(r"Used (\d+) registers", part).group(1))
        spilled = sum(int(x) for x in re.findall(r"(\d+) bytes spill", part))
        out[part.split("'")[0]] = (used, spilled)
    return out


@pytest.fixture(scope="module")
def terms():
    return {k: v for k, v in compiled("learner_terms.cu").items() if "sums_kernel" in k and "PpoOp" in k}


def test_standardised_terms_fit_three_blocks_per_sm(terms):
    """Above two blocks per SM the standardised terms are summed by a form of which an SM holds three, as it does of the plain
    one: a grid of 297 to 444 blocks on 148 SMs is one wave."""
    per_sm = {k: REGISTERS_PER_SM // (-(-regs // 8) * 8 * THREADS) for k, (regs, _) in terms.items()}
    assert len(per_sm) == 3, terms
    assert sorted(per_sm.values())[0] == 2 and sorted(per_sm.values())[1] >= 3, terms


def test_no_spills(terms):
    assert all(spilled == 0 for _, spilled in terms.values()), terms
