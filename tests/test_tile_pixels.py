"""Where a tile stores its pixels: no division by the length of a row where channels are one dense run (no GPU)."""
import os
import re

from paper_2012_09849_b200 import build as hb


def test_dense_outputs_take_no_division():
    text = re.sub(r"//[^\n]*", "", open(os.path.join(hb.PKG, "csrc", "policy_ref.cu")).read())
    stores = [m.end() for m in re.finditer(r"if \(px >= total\) continue;", text)]
    assert len(stores) == 2                              # the tiles' and the latency form's
    for at in stores:
        row = text[at:text.index(";", at)]
        assert re.search(r"i = p\.y_rows \? r / p\.Wo : 0, x = r - i \* p\.Wo", row), row
    # what follows is the same place: row 0 of a dense layout goes on over all rows, and so do planes of one pixel a row
    assert re.search(r"p\.y_rows = yl\.pitch != Wo \|\| yl\.phases != 1;", text) and "c1.s2d = c1.y_rows = true;" in text
