"""Where a tile's block looks its inputs up: no division by the number of a layout's phases (no GPU)."""
import os
import re

from paper_2012_09849_b200 import build as hb


def test_rows_are_found_without_a_division():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(hb.PKG, "csrc", "conv_strip.cuh")).read())
    for name in ("x_row", "x_tap", "y_row"):
        body = re.search(r"__device__ __forceinline__ int " + name + r"\([^{]*\{([^}]*)\}", text).group(1)
        assert not re.search(r"[/%]", body), (name, body)
    # shifts stand for one phase or two: what the layouts have
    for y in range(9):
        for phases in (1, 2):
            assert (y & (phases - 1), y >> (phases - 1)) == (y % phases, y // phases)
    common = open(os.path.join(hb.PKG, "csrc", "common.cuh")).read()
    assert set(re.findall(r"rows_strips\(g\.\w+, g\.\w+, (\d)\)", common)) == {"1", "2"}
