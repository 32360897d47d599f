"""Performance cases: what users of this library have it do, over its real range.

Each case is a dict of plain values.  ``listed()`` gives the fixed ones,
``draw(rng)`` one more of the same ranges, ``prepare(case, seed)`` what a
program holds before the call, ``run(state)`` one pass through the public
entry points, ``work(case)`` the bytes and operations a pass cannot do
without, and ``exact(case, seed)`` the outputs in plain torch.

Inputs are drawn on the device from the seed alone.  Their distributions are
those of ``paper_1803_01237_gb300.inputs`` (uniform, 32 Gaussian clusters,
Zipf duplicates, Plummer-sphere Morton codes, lognormal).
"""
from __future__ import annotations

import random

import numpy as np
import torch

from paper_1803_01237_gb300 import hss

SIGN = -(1 << 63)


def listed():
    return [
        # one small array: the latency of a call, its launches and its host round trips
        {"name": "sort_small", "kind": "sort", "n": 1 << 15, "p": 4, "eps": 0.05, "dist": "uniform",
         "key_type": "u64", "payload": False},
        # a ragged table column with its row numbers: signed keys, many duplicates, odd sizes
        {"name": "sort_ragged_pairs", "kind": "sort", "n": 1000003, "p": 37, "eps": 0.05, "dist": "zipf",
         "key_type": "i64", "payload": True},
        # the benchmark's workload, one case per kind of input
        {"name": "sort_uniform", "kind": "sort", "n": 1 << 28, "p": 1024, "eps": 0.02, "dist": "uniform",
         "key_type": "u64", "payload": False},
        {"name": "sort_clusters", "kind": "sort", "n": 1 << 28, "p": 1024, "eps": 0.02, "dist": "gauss_mix",
         "key_type": "u64", "payload": False},
        {"name": "sort_duplicates", "kind": "sort", "n": 100000007, "p": 1000, "eps": 0.02, "dist": "zipf",
         "key_type": "u64", "payload": False},
        # particles in Morton order with their index, at a large processor count
        {"name": "sort_particles", "kind": "sort", "n": 1 << 28, "p": 4096, "eps": 0.01, "dist": "morton",
         "key_type": "u64", "payload": True},
        # the same particles at the largest processor count, through groups of processors
        {"name": "two_stage_particles", "kind": "two_stage", "n": 1 << 28, "p": 16384, "groups": 128, "eps": 0.01,
         "dist": "morton", "key_type": "u64", "payload": True},
        # partition requests as the server gets them: a small one and one at its largest processor count
        {"name": "partition_request", "kind": "partition", "n": 1 << 20, "p": 256, "eps": 0.02, "dist": "lognormal",
         "key_type": "u64"},
        {"name": "partition_many", "kind": "partition", "n": 1 << 25, "p": 4096, "eps": 0.02, "dist": "lognormal",
         "key_type": "u64"},
        # many independent jobs in one call
        {"name": "batch_jobs", "kind": "batch", "jobs": 1024, "lo_log2": 10, "hi_log2": 20, "plan": 1, "eps": 0.05,
         "key_type": "i64"},
        # host arrays in, host arrays out
        {"name": "sort_host", "kind": "sort_host", "n": 1 << 26, "p": 256, "eps": 0.02, "dist": "uniform",
         "key_type": "u64"},
        # the server's online training of its model of the key distribution
        {"name": "model_train", "kind": "model", "points": 4096, "steps": 20},
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> int:
    return int(lo * (hi / lo) ** rng.random())


def draw(rng: random.Random):
    kind = rng.choice(["sort", "sort", "sort", "sort", "pairs", "pairs", "partition", "partition", "two_stage", "batch",
                       "sort_host", "model"])
    eps = rng.choice([0.01, 0.02, 0.05])
    key_type = rng.choice(["u64", "u64", "i64"])
    dist = rng.choice(["uniform", "gauss_mix", "zipf", "morton", "lognormal"])
    if kind in ("sort", "pairs"):
        n = _log_uniform(rng, 1 << 15, 1 << 27)
        return {"kind": "sort", "n": n, "p": _log_uniform(rng, 4, min(2048, n // 512)), "eps": eps, "dist": dist,
                "key_type": key_type, "payload": kind == "pairs"}
    if kind == "partition":
        n = _log_uniform(rng, 1 << 16, 1 << 26)
        return {"kind": kind, "n": n, "p": _log_uniform(rng, 64, min(4096, n // 128)), "eps": eps, "dist": dist,
                "key_type": key_type}
    if kind == "two_stage":
        groups = _log_uniform(rng, 16, 160)
        per_group = _log_uniform(rng, 16, 160)
        return {"kind": kind, "n": _log_uniform(rng, 1 << 24, 1 << 27), "p": groups * per_group, "groups": groups,
                "eps": eps, "dist": dist, "key_type": key_type, "payload": rng.random() < 0.5}
    if kind == "batch":
        return {"kind": kind, "jobs": _log_uniform(rng, 16, 1024), "lo_log2": 10, "hi_log2": rng.randint(14, 20),
                "plan": rng.randrange(1 << 30), "eps": eps, "key_type": key_type}
    if kind == "sort_host":
        return {"kind": kind, "n": _log_uniform(rng, 1 << 20, 1 << 26), "p": _log_uniform(rng, 16, 512), "eps": eps,
                "dist": rng.choice(["uniform", "zipf"]), "key_type": key_type}
    return {"kind": "model", "points": _log_uniform(rng, 256, 8192), "steps": rng.randint(2, 30)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed: int, stream: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + stream) & ((1 << 62) - 1))
    return g


def _random64(n: int, g: torch.Generator) -> torch.Tensor:
    """n words of 64 random bits."""
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    out.random_(-(1 << 63), None, generator=g)
    return out


def _uniform(n, g):
    return _random64(n, g)


def _gauss_mix(n, g):
    means = _random64(32, g)
    off = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).mul_(2.0 ** 40).round_().to(torch.int64)
    return off.add_(means[torch.randint(0, 32, (n,), device="cuda", generator=g)])


def _zipf_ranks(n, g, distinct, s):
    w = torch.arange(1, distinct + 1, dtype=torch.float64, device="cuda") ** (-s)
    cdf = torch.cumsum(w, 0)
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g).mul_(cdf[-1])
    return torch.searchsorted(cdf, u, right=True).clamp_(max=distinct - 1)


def _zipf(n, g):
    values = _random64(1 << 12, g)
    return values[_zipf_ranks(n, g, 1 << 12, 1.2)]


def _lognormal(n, g):
    x = torch.randn(n, dtype=torch.float64, device="cuda", generator=g).mul_(2.0).sub_(12.0).exp_()
    return x.clamp_(max=1.0).mul_(float((1 << 63) - 1024)).floor_().to(torch.int64)


def _spread3(v):
    v = (v | (v << 32)) & 0x1F00000000FFFF
    v = (v | (v << 16)) & 0x1F0000FF0000FF
    v = (v | (v << 8)) & 0x100F00F00F00F00F
    v = (v | (v << 4)) & 0x10C30C30C30C30C3
    return (v | (v << 2)) & 0x1249249249249249


def _morton(n, g):
    def radius(m):
        return (m ** (-2.0 / 3.0) - 1.0) ** -0.5

    r_max = radius(0.999)
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    chunk = 1 << 26
    for a in range(0, n, chunk):
        m = min(n, a + chunk) - a
        r = radius(0.999 * (1.0 - torch.rand(m, dtype=torch.float64, device="cuda", generator=g)))
        v = torch.randn(3, m, dtype=torch.float64, device="cuda", generator=g)
        v *= r / v.square().sum(0).clamp_(min=1e-24).sqrt_()
        q = ((v + r_max) / (2.0 * r_max) * float(1 << 21)).floor_().clamp_(0, (1 << 21) - 1).to(torch.int64)
        out[a:a + m] = _spread3(q[0]) | (_spread3(q[1]) << 1) | (_spread3(q[2]) << 2)
    return out


DISTRIBUTIONS = {"uniform": _uniform, "gauss_mix": _gauss_mix, "zipf": _zipf, "lognormal": _lognormal,
                 "morton": _morton}


def _keys(case, seed):
    return DISTRIBUTIONS[case["dist"]](case["n"], _gen(seed, 1))


def _job_plan(case):
    """Sizes (log-uniform), processor counts and kinds of a batch's jobs."""
    rng = random.Random(case["plan"])
    lo, hi = case["lo_log2"], case["hi_log2"]
    sizes = [int(2.0 ** (lo + (hi - lo) * rng.random())) for _ in range(case["jobs"])]
    zipf = [rng.random() < 0.5 for _ in sizes]
    return sizes, [max(1, min(n, max(4, n >> 14))) for n in sizes], zipf


def _batch_keys(case, seed):
    """Each job uniform, or Zipf over 2^16 values of its own."""
    sizes, _, zipf = _job_plan(case)
    g = _gen(seed, 2)
    n = sum(sizes)
    keys = _random64(n, g)
    job = torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), torch.tensor(sizes, device="cuda"))
    x = (job << 16) + _zipf_ranks(n, g, 1 << 16, 1.1)
    for mul in (-7046029254386353131, -4658895280553007687):  # odd multipliers: distinct values stay distinct
        x = x * mul
        x = x ^ ((x >> 32) & 0xFFFFFFFF)
    return torch.where(torch.tensor(zipf, device="cuda")[job], x, keys)


def _model_points(case, seed):
    """(keys, ranks) pairs as splitters give them: keys of a lognormal sample
    and their ranks on the trainer's 2^40 scale."""
    n = case["points"]
    k = torch.sort(_lognormal(n, _gen(seed, 3)))[0].contiguous()
    scale = 1 << 40
    ranks = (torch.arange(n, dtype=torch.int64, device="cuda") * scale) // n
    return k, ranks, scale


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    st = {"case": case, "seed": int(seed)}
    kind = case["kind"]
    if kind == "model":
        st["keys"], st["ranks"], st["scale"] = _model_points(case, seed)
        st["init"] = hss.CDFModel().init(3 + int(seed), "log", 1, (1 << 63) - 1)
        st["model"] = hss.CDFModel()
        return st
    if kind == "batch":
        st["sizes"], st["ps"], _ = _job_plan(case)
        st["keys"] = _batch_keys(case, seed)
        st["out"] = torch.empty_like(st["keys"])
        return st
    keys = _keys(case, seed)
    if kind == "sort_host":
        pinned = torch.empty(case["n"], dtype=torch.int64, pin_memory=True)
        pinned.copy_(keys)
        st["pinned"] = (pinned, torch.empty(case["n"], dtype=torch.int64, pin_memory=True))
        st["keys"], st["out"] = (t.numpy().view(np.uint64) if case["key_type"] == "u64" else t.numpy()
                                 for t in st["pinned"])
        return st
    st["keys"] = keys
    if kind != "partition":
        st["out"] = torch.empty_like(keys)
        st["payload"] = st["out_payload"] = None
        if case["payload"]:
            st["payload"] = torch.arange(case["n"], dtype=torch.int32, device="cuda")
            st["out_payload"] = torch.empty_like(st["payload"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "model":
        m = state["model"]
        m.buf.copy_(state["init"].buf)
        loss = m.train(state["keys"], state["ranks"], state["scale"], case["steps"], 0.01)
        return {"theta": m.theta, "loss": loss, "y": m.eval(state["keys"])}
    seed, eps, kt = state["seed"], case["eps"], case["key_type"]
    if kind == "batch":
        r = hss.sort_batch(state["keys"], state["sizes"], state["ps"], eps, seed, key_type=kt, out=state["out"])
        return {"keys": r.keys, "splitters": r.splitters, "offsets": r.offsets}
    if kind == "partition":
        r, ws = hss.partition(state["keys"], case["p"], eps, seed, key_type=kt)
        # the locally sorted keys stay at the start of the workspace
        return {"splitters": r.splitters, "offsets": r.offsets, "local": ws[:8 * case["n"]].view(torch.int64)}
    if kind == "sort_host":
        out, _, spl, off, _ = hss.sort_host(state["keys"], case["p"], eps, seed, key_type=kt, out=state["out"])
        return {"keys": out.view(np.int64), "splitters": spl, "offsets": off.view(np.int64)}
    if kind == "two_stage":
        r = hss.sort_two_stage(state["keys"], case["p"], case["groups"], eps, seed, payload=state["payload"],
                               key_type=kt, out=state["out"], out_payload=state["out_payload"])
        res = {"keys": r.keys, "splitters": r.splitters, "group_splitters": r.group_splitters, "offsets": r.offsets}
    else:
        r = hss.sort(state["keys"], case["p"], eps, seed, payload=state["payload"], key_type=kt, out=state["out"],
                     out_payload=state["out_payload"])
        res = {"keys": r.keys, "splitters": r.splitters, "offsets": r.offsets}
    if r.payload is not None:
        res["payload"] = r.payload
    return res


def work(case):
    kind = case["kind"]
    if kind == "model":
        # 1-32-32-1 network: forward 2 (32 + 1024 + 32), twice that backward, per point and step; one more forward
        n, fwd = case["points"], 2 * (32 + 1024 + 32)
        return {"bytes": 16 * n + 4 * n + 8 * 3 * 1153, "flops": n * fwd * (3 * case["steps"] + 1)}
    if kind == "batch":
        sizes, ps, _ = _job_plan(case)
        return {"bytes": 16 * sum(sizes) + sum(24 * p for p in ps), "flops": 0}
    # every key (and payload) read once and written once, 16 bytes a splitter and 8 an offset
    per_key = 24 if case.get("payload") else 16
    return {"bytes": per_key * case["n"] + 24 * case["p"], "flops": 0}


# ---------------------------------------------------------------------------
# the same outputs in plain torch
# ---------------------------------------------------------------------------
def _sorted(keys, key_type, payload=None):
    flip = SIGN if key_type == "u64" else 0
    k, order = torch.sort(keys ^ flip, stable=True)
    return k ^ flip, (payload[order] if payload is not None else None)


def _exact_model(case, seed):
    keys, ranks, scale = _model_points(case, seed)
    theta = hss.CDFModel().init(3 + int(seed), "log", 1, (1 << 63) - 1).theta.to(torch.float64)
    lo, hi = np.log2(2.0), np.log2(float(1 << 63))
    x = ((torch.log2(1.0 + keys.to(torch.float64)) - lo) / (hi - lo)).clamp(0.0, 1.0)
    t = ranks.to(torch.float64) / scale

    def net(th):
        w1, b1, w2, b2, w3, b3 = torch.split(th, [32, 32, 1024, 32, 32, 1])
        h = torch.relu(x[:, None] * w1 + b1)
        return torch.relu(h @ w2.view(32, 32).T + b2) @ w3 + b3

    m = torch.zeros_like(theta)
    v = torch.zeros_like(theta)
    loss = None
    for k in range(1, case["steps"] + 1):
        th = theta.clone().requires_grad_(True)
        loss = (net(th) - t).square().mean()
        (g,) = torch.autograd.grad(loss, th)
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        theta = theta - 0.01 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return {"theta": theta, "loss": loss.detach().reshape(1), "y": net(theta).detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "model":
        return _exact_model(case, seed)
    if kind == "partition":
        return None
    if kind == "batch":
        keys = _batch_keys(case, seed)
        sizes, _, _ = _job_plan(case)
        out = torch.cat([_sorted(k, case["key_type"])[0] for k in torch.split(keys, sizes)])
        return {"keys": out, "splitters": None, "offsets": None}
    payload = torch.arange(case["n"], dtype=torch.int32, device="cuda") if case.get("payload") else None
    k, pay = _sorted(_keys(case, seed), case["key_type"], payload)
    if kind == "sort_host":
        k = k.cpu().numpy()
    res = {"keys": k, "splitters": None, "offsets": None}
    if kind == "two_stage":
        res["group_splitters"] = None
    if pay is not None:
        res["payload"] = pay
    return res
