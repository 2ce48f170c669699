"""The host-buffer step on both sides of the batch size up to which the kernels use the context's pinned words themselves:
every output against the device step, per-row times, buffers left by a larger and a smaller call."""
import dataclasses

import numpy as np
import pytest

import hts_workloads as wl
import paper_2012_09849_b200 as hts
from gpu_util import Policy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
def test_outputs_are_those_of_the_device_step(dtype):
    cfg = dataclasses.replace(wl.CONFIGS[2], weight_dtype=dtype)
    pol = Policy(cfg, max_batch=300)
    try:
        for n, own_t, logits in ((128, True, True), (300, False, False), (129, True, True), (1, False, True), (127, True, False)):
            obs = wl.make_obs(cfg, n, batch_index=n)
            ids = np.arange(7, 7 + n, dtype=np.int32)
            t = (np.arange(n, dtype=np.int32) * 3) % 11 if own_t else None
            dev = pol.step(obs, ids, 2, 5, t_per_env=t)
            out = {"actions": np.full(n, -1, np.int32), **{k: np.full(n, np.nan, np.float32) for k in ("logp", "values", "entropy")}}
            if logits:
                out["logits"] = np.full((n, cfg.A), np.nan, np.float32)
            hts.hts_policy_step_host(pol.ctx, obs, ids, t, 2, 5, n, out["actions"], out["logp"], out["values"], out["entropy"],
                                     out.get("logits"))
            assert hts.hts_last_async_error(pol.ctx) == 0
            for k, v in out.items():
                assert np.array_equal(v.view(np.int32), dev[k].view(np.int32)), (n, k)
    finally:
        pol.close()
