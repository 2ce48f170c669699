"""A block of a cluster may be written to only once it has started: the order of the operations in the sources (no GPU)."""
import os
import re

import pytest

from paper_2012_09849_b200 import build as hb

# source, kernel, what says that a block has started, what waits for all of them, what reaches into another block
KERNELS = [("learner_terms.cu", "terms_cluster_kernel", "cluster_started(", "cluster_wait(", "store_to_rank("),
           ("fc_tc.cu", "fc_pair_kernel", "cluster_sync(", "cluster_sync(", "in_first(")]


@pytest.mark.parametrize("source,kernel,started,waited,reaches", KERNELS, ids=[k[1] for k in KERNELS])
def test_every_block_has_started_before_another_reaches_into_it(source, kernel, started, waited, reaches):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(hb.PKG, "csrc", source)).read())
    start = text.index(kernel + "(")
    body = text[text.index("{", start):]
    body = body[:body.index("\n}")]
    assert 0 <= body.find(started) <= body.find(waited) < body.find(reaches)
