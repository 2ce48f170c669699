"""What the fp32 path's copying kernels wait for, and when: the order of the operations in the sources (no GPU)."""
import os
import re

import pytest

from paper_2012_09849_b200 import build as hb

KERNELS = [("conv_strip.cu", "conv_strip_kernel"), ("fc_f32.cu", "fc_lanes_kernel")]


def branches(source, kernel):
    """The copying warp's part of a kernel, and the computing warps'."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(hb.PKG, "csrc", source)).read())
    body = text[text.index("{", text.index(kernel + "(")):]
    body = body[:body.index("\n}")]
    start = body.index("if (warp == NC) {")
    end = body.index("\n    }\n", start)
    return body[start:end], body[end:]


@pytest.mark.parametrize("source,kernel", KERNELS, ids=[k[1] for k in KERNELS])
def test_the_limit_of_a_wait_does_not_count_the_kernel_before(source, kernel):
    for part in branches(source, kernel):
        assert 0 <= part.find("pdl_wait()") < part.find("mbar_wait_warp(")


@pytest.mark.parametrize("source,kernel", KERNELS, ids=[k[1] for k in KERNELS])
def test_copies_in_flight_land_before_a_warp_that_gave_up_goes_on(source, kernel):
    """A wait after one that gave up ends at once, landed or not: what follows must be time, not a wait."""
    copies, computes = branches(source, kernel)
    assert "mbar_wait_warp(full" not in copies
    assert copies.rstrip().endswith("if (st < stages) tc::let_copies_land();\n        return;")
    gives_up = re.search(r"if \(!tc::mbar_wait_warp\(full[^{;]*\{\s*tc::let_copies_land\(\);\s*break;", computes)
    assert gives_up and computes.count("mbar_wait_warp(") == 1
