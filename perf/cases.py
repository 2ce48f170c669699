"""The framework's work as cases: what a synchronous actor-critic run has it do, through its public entry points.

Kinds of pass, and the calls each makes
  actor       hts_policy_step: frames on the device, dense
  executor    hts_policy_step_indexed: frames gathered by slot from the state buffer, outputs scattered into a row of the storage
  host        hts_policy_step_host: frames and results in pinned host memory, copies inside the call
  advantages  hts_gae over the [T, N] storage
  vtrace      hts_vtrace over the [T, N] storage
  terms       hts_a2c_terms / hts_ppo_terms over the storage
  update      one learner update: hts_policy_evaluate, the terms, hts_policy_gradient, hts_policy_load_weights of the
              learner, hts_delayed_update of the parameters, hts_policy_load_weights of the actor

Shapes are those of the five configurations in hts_workloads.py (4x84x84 and 16x72x96 frames); drawn cases also take two of the
other frame shapes that the tests run.  Batches go from one observation to the whole pool of 8192 environments.
"""
import math

import torch

import paper_2012_09849_b200 as hts

FRAMES = {"atari": (4, 84, 84), "football": (16, 72, 96), "wide": (4, 64, 96), "eight": (8, 84, 84)}
GAMMA, LAM = 0.99, 0.95
DTYPES = {"fp32": (hts.HTS_DTYPE_FP32, torch.float32), "bf16": (hts.HTS_DTYPE_BF16, torch.bfloat16)}


def listed():
    return [
        # the tiny actor-critic configuration: 16 environments, fp32 network, every step of a rollout is one such call
        {"name": "actor-fp32-16", "kind": "actor", "frames": "atari", "actions": 6, "dtype": "fp32", "n": 16, "own_t": False},
        # actor-critic with 256 environments: launch latency of the five-layer chain
        {"name": "actor-256", "kind": "actor", "frames": "atari", "actions": 18, "dtype": "bf16", "n": 256, "own_t": False},
        # proximal policy optimisation with 1024 environments: the headline actor step
        {"name": "actor-1024", "kind": "actor", "frames": "atari", "actions": 18, "dtype": "bf16", "n": 1024, "own_t": False},
        # football minimaps: 16 sparse planes, 512 environments
        {"name": "actor-football-512", "kind": "actor", "frames": "football", "actions": 19, "dtype": "bf16", "n": 512, "own_t": False},
        # an asynchronous executor batch: a ragged random subset of the 8192-environment pool, each at its own time step
        {"name": "executor-1733-of-8192", "kind": "executor", "frames": "atari", "actions": 18, "dtype": "bf16", "n": 1733, "pool": 8192, "own_t": True},
        # the whole pool in one batch: throughput
        {"name": "actor-8192", "kind": "actor", "frames": "atari", "actions": 18, "dtype": "bf16", "n": 8192, "own_t": False},
        # simulators on the host: frames come from pinned memory and the actions go back to it
        {"name": "host-1024", "kind": "host", "frames": "atari", "actions": 18, "dtype": "bf16", "n": 1024, "own_t": False},
        # the advantage scan that closes a 128-step rollout of 1024 environments
        {"name": "advantages-128x1024", "kind": "advantages", "T": 128, "N": 1024, "p_done": 0.005},
        # the off-policy-corrected scan over a long football rollout
        {"name": "vtrace-512x512", "kind": "vtrace", "T": 512, "N": 512, "p_done": 0.002},
        # the clipped objective's sample means over a whole 128 x 1024 storage
        {"name": "terms-ppo-131072", "kind": "terms", "objective": "ppo", "normalize": True, "count": 131072},
        # one actor-critic update on the 5 x 16 transitions of the tiny configuration
        {"name": "update-a2c-80", "kind": "update", "objective": "a2c", "frames": "atari", "actions": 6, "n": 80},
        # one minibatch of the proximal policy optimisation learner
        {"name": "update-ppo-1024", "kind": "update", "objective": "ppo", "frames": "atari", "actions": 18, "n": 1024},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["actor", "actor", "actor", "executor", "host", "advantages", "vtrace", "terms", "update", "update"])
    if kind in ("advantages", "vtrace"):
        T = _log(rng, 1, 512)
        return {"kind": kind, "T": T, "N": _log(rng, 16, min(1 << 17, (1 << 24) // T)), "p_done": rng.choice([0.002, 0.005, 0.02])}
    if kind == "terms":
        return {"kind": kind, "objective": rng.choice(["a2c", "ppo"]), "normalize": rng.random() < 0.5, "count": _log(rng, 64, 1 << 24)}
    frames = rng.choice(["atari", "atari", "atari", "football", "football", "wide", "eight"])
    case = {"kind": kind, "frames": frames, "actions": rng.choice([6, 18, 19, rng.randint(2, 32)])}
    if kind == "update":
        return {**case, "objective": rng.choice(["a2c", "ppo"]), "n": _log(rng, 5, 512 if frames == "football" else 1000)}
    case["own_t"] = rng.random() < 0.5
    case["dtype"] = "fp32" if rng.random() < 0.25 else "bf16"
    most = 1024 if case["dtype"] == "fp32" else 2048 if kind == "host" else 8192
    case["n"] = _log(rng, 1, most)
    if kind == "executor":
        case["pool"] = _log(rng, case["n"], 8192)
    return case


class _Context:
    """An hts context with its weights loaded, destroyed with its last reference."""

    def __init__(self, frames, actions, dtype, max_batch, weights):
        self.handle = hts.hts_policy_create(*frames, actions, DTYPES[dtype][0], max_batch)
        hts.hts_policy_load_weights(self.handle, weights)

    def __del__(self):
        if getattr(self, "handle", None):
            hts.hts_policy_destroy(self.handle)


def _shapes(frames, actions):
    c, h, w = frames
    for k, s in ((8, 4), (4, 2), (3, 1)):
        h, w = (h - k) // s + 1, (w - k) // s + 1
    return {"conv1_w": (32, c, 8, 8), "conv1_b": (32,), "conv2_w": (64, 32, 4, 4), "conv2_b": (64,), "conv3_w": (64, 64, 3, 3),
            "conv3_b": (64,), "fc_w": (512, 64 * h * w), "fc_b": (512,), "pi_w": (actions, 512), "pi_b": (actions,),
            "v_w": (1, 512), "v_b": (1,)}


def _macs(frames, actions):
    """Multiply-adds of one observation: (first convolution, whole network)."""
    c, h, w = frames
    per, first = 0, 0
    for cin, cout, k, s in ((c, 32, 8, 4), (32, 64, 4, 2), (64, 64, 3, 1)):
        h, w = (h - k) // s + 1, (w - k) // s + 1
        per += h * w * cout * cin * k * k
        first = first or per
    return first, per + 64 * h * w * 512 + 512 * (actions + 1)


def _views(flat, shapes):
    """The parameter tensors as consecutive views of one flat buffer, the layout hts_delayed_update is called on."""
    out, at = {}, 0
    for name, shape in shapes.items():
        size = math.prod(shape)
        out[name] = flat[at:at + size].view(shape)
        at += size
    return out


def _flat_weights(shapes, g):
    """He-normal weights, uniform biases."""
    flat = torch.empty(sum(math.prod(s) for s in shapes.values()), device="cuda")
    for name, view in _views(flat, shapes).items():
        if name.endswith("_w"):
            view.normal_(0.0, math.sqrt(2.0 / math.prod(view.shape[1:])), generator=g)
        else:
            view.uniform_(-0.1, 0.1, generator=g)
    return flat


def _frames(case, n, g):
    """uint8 pixels: uniform for video frames, 255 with probability 0.02 for minimaps."""
    shape = (n, *FRAMES[case["frames"]])
    if case["frames"] == "football":
        return (torch.randint(0, 50, shape, dtype=torch.uint8, device="cuda", generator=g) == 0).to(torch.uint8) * 255
    return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=g)


def _prepare_step(case, seed, g):
    frames, A, n = FRAMES[case["frames"]], case["actions"], case["n"]
    flat = _flat_weights(_shapes(frames, A), g).to(DTYPES[case["dtype"]][1])
    s = {"case": case, "n": n, "seed": seed * 0x9E3779B97F4A7C15 % (1 << 64)}
    s["ctx"] = _Context(frames, A, case["dtype"], n, _views(flat, _shapes(frames, A)))
    rows = case.get("pool", n)
    obs = _frames(case, rows, g)
    ids = torch.randperm(65536, device="cuda", generator=g)[:n].to(torch.int32)
    t = torch.randint(0, 128, (n,), dtype=torch.int32, device="cuda", generator=g) if case["own_t"] else None
    s["slots"] = torch.randperm(rows, device="cuda", generator=g)[:n].to(torch.int32)
    out = [torch.zeros(rows, dtype=d, device="cuda") for d in (torch.int32, torch.float32, torch.float32, torch.float32)]
    if case["kind"] == "host":
        obs, ids, t = (None if x is None else x.cpu().pin_memory() for x in (obs, ids, t))
        out = [x.cpu().pin_memory() for x in out]
    s.update(obs=obs, ids=ids, t=t, out=out)
    return s


def _prepare_scan(case, g):
    T, N = case["T"], case["N"]
    uniform = torch.rand(T, N, device="cuda", generator=g)
    normal = [torch.randn(T, N, device="cuda", generator=g) for _ in range(2)]
    s = {"case": case, "rewards": torch.sign(normal[1]) * (uniform < 0.03), "values": normal[0]}
    s["dones"] = (torch.rand(T, N, device="cuda", generator=g) < case["p_done"]).to(torch.uint8)
    s["bootstrap"] = torch.randn(N, device="cuda", generator=g)
    if case["kind"] == "vtrace":
        s["log_rhos"] = 0.3 * torch.randn(T, N, device="cuda", generator=g)
    s["out"] = [torch.empty(T, N, device="cuda") for _ in range(2)]
    return s


def _prepare_terms(case, g):
    count = case["count"]
    x = {k: torch.randn(count, device="cuda", generator=g) for k in ("values", "advantages", "returns")}
    x["logp"] = -3.0 * torch.rand(count, device="cuda", generator=g)
    x["logp_old"] = x["logp"] + 0.1 * torch.randn(count, device="cuda", generator=g)
    x["entropy"] = 2.9 * torch.rand(count, device="cuda", generator=g)
    return {"case": case, **x, "out": torch.empty(3 if case["objective"] == "a2c" else 4, device="cuda")}


def _prepare_update(case, g):
    frames, A, n = FRAMES[case["frames"]], case["actions"], case["n"]
    shapes = _shapes(frames, A)
    before = _flat_weights(shapes, g)                      # the parameters the rollout was collected with
    theta = before + 1e-4 * torch.randn(before.numel(), device="cuda", generator=g)
    s = {"case": case, "n": n, "theta": theta, "grad": torch.zeros_like(theta), "half": theta.to(torch.bfloat16)}
    s["sq"] = 1e-4 * torch.rand(theta.numel(), device="cuda", generator=g)
    for name, flat in (("w_theta", theta), ("w_grad", s["grad"]), ("w_half", s["half"])):
        s[name] = _views(flat, shapes)
    s["learner"] = _Context(frames, A, "fp32", n, _views(before, shapes))
    s["actor"] = _Context(frames, A, "bf16", 16, s["w_half"])
    s["obs"] = _frames(case, n, g)
    s["actions"] = torch.randint(0, A, (n,), dtype=torch.int32, device="cuda", generator=g)
    s["advantages"], s["returns"] = (torch.randn(n, device="cuda", generator=g) for _ in range(2))
    s["logp"], s["values"], s["entropy"] = (torch.empty(n, device="cuda") for _ in range(3))
    s["terms"] = torch.empty(3 if case["objective"] == "a2c" else 4, device="cuda")
    s["logp_old"] = None
    if case["objective"] == "ppo":                         # an earlier epoch of the same storage: the ratios have moved
        s["logp_old"] = torch.empty(n, device="cuda")
        hts.hts_policy_evaluate(s["learner"].handle, s["obs"], s["actions"], n, s["logp_old"], s["values"], s["entropy"])
        s["logp_old"] += 0.15 * torch.randn(n, device="cuda", generator=g)
    return s


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    if kind in ("actor", "executor", "host"):
        return _prepare_step(case, seed, g)
    if kind in ("advantages", "vtrace"):
        return _prepare_scan(case, g)
    return _prepare_terms(case, g) if kind == "terms" else _prepare_update(case, g)


def _run_update(s):
    n, learner, ppo = s["n"], s["learner"].handle, s["logp_old"] is not None
    clip = 0.2 if ppo else 0.0
    hts.hts_policy_evaluate(learner, s["obs"], s["actions"], n, s["logp"], s["values"], s["entropy"])
    if ppo:
        hts.hts_ppo_terms(s["logp"], s["logp_old"], s["values"], s["entropy"], s["advantages"], s["returns"], n, clip, False, s["terms"])
    else:
        hts.hts_a2c_terms(s["logp"], s["values"], s["entropy"], s["returns"], n, s["terms"])
    hts.hts_policy_gradient(learner, s["obs"], s["actions"], s["advantages"], s["returns"], s["logp_old"], 0.5, 0.01, clip, n, s["w_grad"])
    # the next gradient is taken at the parameters this update starts from (one-step delay)
    hts.hts_policy_load_weights(learner, s["w_theta"])
    # a step size late in its decay: the same storage is used by every pass
    hts.hts_delayed_update(s["theta"], s["grad"], s["sq"], s["theta"].numel(), 1e-5, 0.99, 1e-5, s["half"])
    hts.hts_policy_load_weights(s["actor"].handle, s["w_half"])
    return {"grads": s["w_grad"], "theta": s["theta"], "sq": s["sq"], "half": s["half"], "terms": s["terms"], "logp": s["logp"],
            "values": s["values"], "entropy": s["entropy"]}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "update":
        return _run_update(s)
    out = s["out"]
    if kind == "actor":
        hts.hts_policy_step(s["ctx"].handle, s["obs"], s["ids"], s["t"], 3, s["seed"], s["n"], *out)
    elif kind == "executor":
        hts.hts_policy_step_indexed(s["ctx"].handle, s["obs"], case["pool"], s["slots"], s["ids"], s["t"], 3, s["seed"], s["n"], *out)
    elif kind == "host":
        hts.hts_policy_step_host(s["ctx"].handle, s["obs"], s["ids"], s["t"], 3, s["seed"], s["n"], *out)
    elif kind == "advantages":
        hts.hts_gae(s["rewards"], s["values"], s["dones"], s["bootstrap"], GAMMA, LAM, case["T"], case["N"], *out)
    elif kind == "vtrace":
        hts.hts_vtrace(s["log_rhos"], s["rewards"], s["values"], s["dones"], s["bootstrap"], GAMMA, LAM, 1.0, 1.0, case["T"], case["N"], *out)
    elif case["objective"] == "a2c":
        hts.hts_a2c_terms(s["logp"], s["values"], s["entropy"], s["returns"], case["count"], out)
    else:
        hts.hts_ppo_terms(s["logp"], s["logp_old"], s["values"], s["entropy"], s["advantages"], s["returns"], case["count"], 0.2,
                          case["normalize"], out)
    return out


def work(case):
    kind = case["kind"]
    if kind in ("advantages", "vtrace"):
        # per element: rewards, values, dones and two outputs (and the log ratios); the recurrences of one step
        per = (17, 8) if kind == "advantages" else (21, 20)
        return {"bytes": per[0] * case["T"] * case["N"] + 4 * case["N"], "flops": per[1] * case["T"] * case["N"]}
    if kind == "terms":
        return {"bytes": (16 if case["objective"] == "a2c" else 24) * case["count"], "flops": 20 * case["count"]}
    frames, A, n = FRAMES[case["frames"]], case["actions"], case["n"]
    first, all_layers = _macs(frames, A)
    params = sum(math.prod(s) for s in _shapes(frames, A).values())
    pixels = math.prod(frames) * n
    if kind == "update":
        # evaluation, the gradient's own forward pass, weight gradients, data gradients (none for the frames);
        # parameters and squared averages read and written, gradients and the bf16 copy written
        flops = 2 * n * (4 * all_layers - first)
        return {"bytes": pixels + 36 * n + (4 * 4 + 4 + 2) * params, "flops": flops}
    weights = params * (4 if case["dtype"] == "fp32" else 2)
    index = 4 * n * (1 + bool(case["own_t"]) + (kind == "executor"))
    return {"bytes": pixels + weights + index + 16 * n, "flops": 2 * n * all_layers}


def tolerance(case):
    kind = case["kind"]
    if kind in ("advantages", "vtrace"):
        return {"rel": 1e-5, "max": 1e-4}
    if kind == "terms":
        return {"rel": 1e-5}
    if kind == "update":
        # fp32 sums through four layers and back, a few ReLU decisions at rounding distance; "max" is one last place of
        # the bf16 copy of a parameter
        return {"rel": 5e-5, "max": 1e-2}
    if case["dtype"] == "fp32":
        return {"rel": 2e-5, "differ": 2e-3}
    # bf16 weights and 16-bit activations; a few sampled actions fall the other way (and with them their log-probability)
    return {"rel": 1e-2, "max": 0.9, "differ": 5e-3}
