"""Contexts are independent across threads, also where several make a kernel's first launch at once with shared memory of
different sizes: a process of its own, in which nothing has been launched before."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = """
import dataclasses, threading
import numpy as np, torch
import hts_workloads as wl, paper_2012_09849_b200 as hts

def work(C, H, W, A, dtype, n, start=None):
    cfg = dataclasses.replace(wl.CONFIGS[2], C=C, H=H, W=W, A=A, weight_dtype=dtype)
    dt = hts.HTS_DTYPE_FP32 if dtype == "fp32" else hts.HTS_DTYPE_BF16
    weights = hts.weights_to_device(wl.make_weights(cfg), dt)
    obs = torch.from_numpy(wl.make_obs(cfg, n)).cuda()
    ids = torch.arange(n, dtype=torch.int32, device="cuda")
    act = torch.zeros(n, dtype=torch.int32, device="cuda")
    f = [torch.zeros(n, device="cuda") for _ in range(3)]
    grads = {k: torch.zeros(v.shape, device="cuda") for k, v in weights.items()}
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    ctx = hts.hts_policy_create(C, H, W, A, dt, n)
    if start is not None:
        start.wait()
    with torch.cuda.stream(s):
        hts.hts_policy_load_weights(ctx, weights)
        hts.hts_policy_step(ctx, obs, ids, None, 3, 17, n, act, *f)
        if dtype == "fp32":
            hts.hts_policy_gradient(ctx, obs, act, f[0], f[1], None, 0.5, 0.01, 0.0, n, grads)
    s.synchronize()
    assert hts.hts_last_async_error(ctx) == 0
    hts.hts_policy_destroy(ctx)
    return [x.cpu().numpy() for x in (act, *f, *grads.values())]

CASES = [(4, 84, 84, 6, "fp32", 8), (4, 84, 84, 64, "fp32", 40), (4, 84, 84, 18, "fp32", 120), (4, 84, 84, 64, "bf16", 9),
         (4, 36, 44, 2, "bf16", 30), (16, 72, 96, 19, "bf16", 7), (8, 84, 84, 40, "bf16", 5)]
out, start = [None] * len(CASES), threading.Barrier(len(CASES), timeout=120)
def run(i):
    try:
        out[i] = work(*CASES[i], start=start)
    except Exception as e:
        out[i] = e
threads = [threading.Thread(target=run, args=(i,)) for i in range(len(CASES))]
for t in threads: t.start()
for t in threads: t.join()
for c, o in zip(CASES, out):
    assert isinstance(o, list), (c, o)
    for a, b in zip(o, work(*c)):
        assert np.array_equal(a.view(np.int32), b.view(np.int32)), c
print("same")
"""


def test_first_launches_in_several_threads():
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stdout + r.stderr
