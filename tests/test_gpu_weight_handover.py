"""Launch order around a weight load: the first layer's prologue loads filters and biases, so its launch may overlap the
end of an earlier step but not the kernel that packs them.  Nothing is executed: steps are recorded into a CUDA graph and
its edges are read."""
import ctypes
import dataclasses

import pytest
import torch

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


def programmatic_edges(record):
    """Of the chain of kernels that `record` enqueues: for each but the first, whether it may start before its predecessor ends."""
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g):
        record()
    cu = ctypes.CDLL("libcuda.so.1")
    graph, count = ctypes.c_void_p(int(g.raw_cuda_graph())), ctypes.c_size_t()
    assert cu.cuGraphGetEdges_v2(graph, None, None, None, ctypes.byref(count)) == 0
    n = count.value
    src, dst, data = (ctypes.c_void_p * n)(), (ctypes.c_void_p * n)(), (ctypes.c_ubyte * (8 * n))()
    assert cu.cuGraphGetEdges_v2(graph, src, dst, data, ctypes.byref(count)) == 0
    after = {s: (d, data[8 * i + 2] == 1) for i, (s, d) in enumerate(zip(src, dst))}      # bytes: from port, to port, type
    assert len(after) == n, "one chain"
    node, out = (set(after) - set(dst)).pop(), []
    while node in after:
        node, early = after[node]
        out.append(early)
    return out


@pytest.mark.parametrize("config,n,kernels", [(2, 3, 3), (2, 900, 5), (4, 5, 5)])     # one kernel for the convolutions, three, 16 channels
def test_first_step_after_a_load_waits_for_the_packed_weights(config, n, kernels):
    cfg = dataclasses.replace(wl.CONFIGS[config], N=n)
    pol = Policy(cfg, max_batch=n)
    try:
        obs = torch.zeros(n, cfg.C, cfg.H, cfg.W, dtype=torch.uint8, device="cuda")
        ids = torch.arange(n, dtype=torch.int32, device="cuda")
        out = [torch.zeros(n, dtype=d, device="cuda") for d in (torch.int32, torch.float32, torch.float32, torch.float32)]
        step = lambda: hts.hts_policy_step(pol.ctx, obs, ids, None, 0, 1, n, *out)
        load = lambda: hts.hts_policy_load_weights(pol.ctx, pol.dev_w)
        rest = [True] * (kernels - 1)

        def twice():
            load(); step(); step()
        assert programmatic_edges(twice) == [True, False] + rest + [True] + rest       # largest magnitudes, packing, two steps
        # a load outside of a graph: neither the graph's steps nor the step that follows the load may overlap it
        load()
        assert programmatic_edges(lambda: (step(), step())) == rest + [False] + rest
        step()
        assert programmatic_edges(lambda: (step(), step())) == rest + [True] + rest
        torch.cuda.synchronize()
        assert hts.hts_last_async_error(pol.ctx) == 0
    finally:
        pol.close()
