"""Host steps whose frames are copied in two parts: outputs and hidden layers are those of the device step, bit for bit."""
import ctypes
import dataclasses

import numpy as np
import pytest

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("C,H,W,dtype,sizes", [
    (4, 84, 84, "bf16", (255, 256, 511, 512, 1024, 2500)),        # parts in different kernels: stack and layers, forms of the dense layer
    (16, 72, 96, "bf16", (257, 530)),
    (4, 36, 44, "bf16", (2226, 2227, 2600)),                      # the line lies between the first two
    (4, 36, 44, "fp32", (511, 512, 901))])
def test_outputs_and_layers(C, H, W, dtype, sizes):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W, weight_dtype=dtype)
    pol = Policy(cfg, max_batch=max(sizes) + 5)
    try:
        for n in sizes:
            obs = wl.make_obs(cfg, n, batch_index=n)
            ids, t = np.arange(7, 7 + n, dtype=np.int32), (np.arange(n, dtype=np.int32) * 3) % 11
            dev = pol.step(obs, ids, 2, 5, t_per_env=t)
            layers = [pol.activation(k, n) for k in (1, 2, 3, 4)]
            pol.step(obs[::-1], ids, 2, 5, t_per_env=t)            # other contents in the workspaces
            out = {"actions": np.full(n, -1, np.int32), "logits": np.full((n, cfg.A), np.nan, np.float32),
                   **{k: np.full(n, np.nan, np.float32) for k in ("logp", "values", "entropy")}}
            hts.hts_policy_step_host(pol.ctx, obs, ids, t, 2, 5, n, out["actions"], out["logp"], out["values"], out["entropy"], out["logits"])
            assert hts.hts_last_async_error(pol.ctx) == 0
            for k, v in out.items():
                assert np.array_equal(v.view(np.int32), dev[k].view(np.int32)), (n, k)
            for k, ref in enumerate(layers):
                assert np.array_equal(pol.activation(k + 1, n).view(np.int32), ref.view(np.int32)), (n, "layer", k + 1)
    finally:
        pol.close()


@pytest.mark.parametrize("C,H,W,cut,whole", [
    (4, 36, 44, (2227, 2600), (256, 512, 1105, 2226)),            # few bytes: no step hides behind the second part's copy
    (4, 84, 84, (256, 512), (248, 255)),
    (16, 72, 96, (256,), (64, 255))])                             # few rows: their step is one observation's latency
def test_parts_by_bytes_and_rows(C, H, W, cut, whole):
    """Frames are copied in two parts, each with a step of its own, from 256 rows and 5.2 MB and 4 KB a row on."""
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W)
    pol = Policy(cfg, max_batch=max(cut))
    try:
        for n in cut + whole:
            obs = np.zeros((n, C, H, W), np.uint8)
            ids = np.arange(n, dtype=np.int32)
            out = [np.empty(n, d) for d in (np.int32, np.float32, np.float32, np.float32)]
            before = hts.hts_launch_count()
            hts.hts_policy_step_host(pol.ctx, obs, ids, None, 0, 5, n, *out)
            assert (hts.hts_launch_count() - before > 5) == (n in cut), n      # a step is three or five kernels
    finally:
        pol.close()


def _next_stream_id():
    """Streams of a process are numbered as they are made."""
    cuda, s, i = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_ulonglong()
    assert cuda.cuStreamCreate(ctypes.byref(s), 1) == 0 and cuda.cuStreamGetId(s, ctypes.byref(i)) == 0
    assert cuda.cuStreamDestroy_v2(s) == 0
    return i.value


@pytest.mark.parametrize("dtype,max_batch,made", [("bf16", 256, 1), ("bf16", 255, 0), ("fp32", 512, 1), ("fp32", 511, 0)])
def test_no_call_makes_a_stream(dtype, max_batch, made):
    """The stream of the copies is made with the context, and only if its batches can be cut."""
    cfg = dataclasses.replace(wl.CONFIGS[2], weight_dtype=dtype)
    assert _next_stream_id() + 1 == _next_stream_id()
    before = _next_stream_id()
    pol = Policy(cfg, max_batch=max_batch)
    try:
        created = _next_stream_id()
        assert created - before == 1 + made
        out = [np.empty(max_batch, d) for d in (np.int32, np.float32, np.float32, np.float32)]
        hts.hts_policy_step_host(pol.ctx, np.zeros((max_batch, cfg.C, cfg.H, cfg.W), np.uint8), np.arange(max_batch, dtype=np.int32), None, 0, 5,
                                 max_batch, *out)
        assert _next_stream_id() - created == 1
    finally:
        pol.close()
