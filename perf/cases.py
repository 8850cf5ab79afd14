"""Representative calls of the framework, for timing it over its range of use.

A case is one call a user makes: a single count (smallest to largest, on each
arithmetic path), a group of counts, a sliced count, a persistent batch, and
the learned scorer's training step and inference.  Formulas are the
repository's own workloads (#Cubic-Vertex-Cover, monotone 1-in-3).

A single formula's cost depends on its graph by orders of magnitude, so in the
single, group and sliced cases the graph (hence the plan) belongs to the case
and the seed draws the weights of the clauses (a weighted count: every allowed
assignment of a clause weighs 1..9).  In the batches, whose cost averages over
many formulas, the seed draws the formulas themselves.
"""
import math
import random

import numpy as np
import torch

from paper_1805_00475_gb300 import instances as I
from paper_1805_00475_gb300 import tnc

# primes just below 2^31: allowed by the 30-bit paths beside the default ones,
# and reduced by the general (Barrett) step
WIDE_PRIMES = (2147483647, 2147483629, 2147483587, 2147483579, 2147483563, 2147483549)


def listed():
    return [
        # the smallest count a user asks for: latency of one call
        {"name": "count_1in3_n20", "kind": "count", "problem": "1in3", "n": 20, "m": 12, "graph": 0, "open": 0,
         "path": "int64", "R": 1, "wide": False, "planner": "bisect"},
        # one formula of the batched size, counted alone
        {"name": "count_vc_n60", "kind": "count", "problem": "vc", "n": 60, "m": 0, "graph": 0, "open": 0,
         "path": "int64", "R": 4, "wide": False, "planner": "best"},
        # an open network (counts for every value of 8 variables) modulo the caller's own primes
        {"name": "count_open_vc_n90", "kind": "count", "problem": "vc", "n": 90, "m": 0, "graph": 1, "open": 8,
         "path": "int64", "R": 3, "wide": True, "planner": "best"},
        # a larger formula on the default path
        {"name": "count_vc_n140", "kind": "count", "problem": "vc", "n": 140, "m": 0, "graph": 0, "open": 0,
         "path": "int64", "R": 4, "wide": False, "planner": "best"},
        # 30-bit residues on the tensor cores
        {"name": "count_tc_vc_n160", "kind": "count", "problem": "vc", "n": 160, "m": 0, "graph": 1, "open": 0,
         "path": "tc", "R": 4, "wide": False, "planner": "best"},
        # the largest single counts: 180 vertices, 20 primes <= 251 on the tensor cores
        {"name": "count_p8_vc_n180", "kind": "count", "problem": "vc", "n": 180, "m": 0, "graph": 9, "open": 0,
         "path": "tc_p8", "R": 20, "wide": False, "planner": "best"},
        # uneven 1-in-3 formulas too heavy for the batch, contracted as groups
        {"name": "many_1in3_p8", "kind": "many", "count": 48, "master": 7, "n_lo": 100, "n_hi": 150,
         "path": "tc_p8", "R": 8},
        # a count whose network is cut into 4 slices to bound its memory
        {"name": "sliced_p8_vc_n160", "kind": "sliced", "n": 160, "graph": 1, "slices_log2": 2, "path": "tc_p8",
         "R": 18},
        # the persistent batch on resident descriptors: the throughput workload
        {"name": "batch_vc_n60", "kind": "batch", "problem": "vc", "n": 60, "count": 2048, "R": 4, "upload": False},
        # a batch of uneven light 1-in-3 formulas with its upload in the pass
        {"name": "batch_1in3", "kind": "batch", "problem": "1in3", "n": 80, "count": 777, "R": 2, "upload": True},
        # one training step of the learned edge scorer (forward, backward, Adam) at the training batch
        {"name": "mlp_step_2048", "kind": "mlp_step", "rows": 2048},
        # the scorer's inference for one merge round of 256 formulas with 8 candidates
        {"name": "mlp_infer_2048", "kind": "mlp_infer", "rows": 2048},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["count_int64", "count_int64", "count_tc", "count_p8", "count_p8", "many", "sliced", "batch",
                       "batch", "mlp_step", "mlp_infer"])
    g = rng.randrange(1000)
    if kind == "count_int64":
        wide = rng.random() < 0.3
        if rng.random() < 0.3:
            n = _log_uniform(rng, 9, 70)
            return {"kind": "count", "problem": "1in3", "n": n, "m": max(2, round(n * rng.uniform(0.5, 0.7))), "graph": g,
                    "open": rng.choice([0, 0, 1, 3]), "path": "int64", "R": rng.randint(1, 5), "wide": wide,
                    "planner": "bisect"}
        return {"kind": "count", "problem": "vc", "n": 2 * _log_uniform(rng, 5, 65), "m": 0, "graph": g,
                "open": rng.choice([0, 0, 0, 1, 5]), "path": "int64", "R": rng.randint(1, 6), "wide": wide,
                "planner": "best"}
    if kind == "count_tc":
        return {"kind": "count", "problem": "vc", "n": 2 * rng.randint(45, 70), "m": 0, "graph": g, "open": 0,
                "path": "tc", "R": rng.randint(1, 5), "wide": rng.random() < 0.2, "planner": "best"}
    if kind == "count_p8":
        return {"kind": "count", "problem": "vc", "n": 2 * rng.randint(45, 80), "m": 0, "graph": g, "open": 0,
                "path": "tc_p8", "R": rng.randint(5, 20), "wide": False, "planner": "best"}
    if kind == "many":
        lo = rng.randint(80, 110)
        return {"kind": "many", "count": rng.randint(3, 48), "master": g, "n_lo": lo, "n_hi": lo + rng.randint(10, 35),
                "path": "tc_p8", "R": rng.randint(6, 9)}
    if kind == "sliced":
        return {"kind": "sliced", "n": 2 * rng.randint(50, 75), "graph": g, "slices_log2": rng.randint(1, 3),
                "path": "tc_p8", "R": rng.randint(10, 18)}
    if kind == "batch":
        problem = rng.choice(["vc", "1in3"])
        n = 2 * rng.randint(15, 32) if problem == "vc" else rng.randint(30, 90)
        return {"kind": "batch", "problem": problem, "n": n, "count": _log_uniform(rng, 5, 2000),
                "R": rng.randint(1, 5), "upload": rng.random() < 0.5}
    return {"kind": kind, "rows": _log_uniform(rng, 9, 9000 if kind == "mlp_step" else 70000)}


# ---------------------------------------------------------------- formulas

def _formula(case):
    if case["problem"] == "vc":
        f = I.cubic_vertex_cover(case["n"], case["graph"])
    else:
        f = I.one_in_three(case["n"], case["m"], case["graph"])
    if case["open"]:
        f.open_vars = sorted(random.Random(case["graph"]).sample(range(f.n_vars), case["open"]))
    return f


def _weighted(f, rng):
    """The formula with a weight of 1..9 on every allowed assignment of a clause."""
    tables = []
    for vs, kind in zip(f.clauses, f.kinds):
        allowed = [(bin(i).count("1") == 1) if kind == I.KIND_1IN3 else i != 0 for i in range(1 << len(vs))]
        tables.append([rng.randint(1, 9) if a else 0 for a in allowed])
    return I.Formula(f.n_vars, f.clauses, [I.KIND_TABLE] * len(f.clauses), tables, open_vars=list(f.open_vars))


def _many_formulas(case):
    return I.batch_one_in_three(case["count"], case["master"], case["n_lo"], case["n_hi"], 0.55, 0.72)


def _primes(case):
    return list(WIDE_PRIMES[:case["R"]]) if case.get("wide") else None


def _batch_formulas(case, seed, count):
    if case["problem"] == "vc":
        return [I.cubic_vertex_cover(case["n"], I.derive_seed(seed, i)) for i in range(count)]
    return I.batch_one_in_three(count, seed, max(20, case["n"] * 5 // 8), case["n"], 0.5, 0.65)


def _batch_plans(case, seed):
    """The case's number of light plans: the batch takes these, a heavier formula is counted in a group."""
    tries = case["count"]
    while True:
        tries += tries // 8 + 2
        plans = tnc.plan_many(_batch_formulas(case, seed, tries), heuristic="best", rank_cap=64)
        light = [p for p in plans if p.stats.max_rank <= 16 and p.stats.total_macs <= 2.0 ** 24]
        if len(light) >= case["count"]:
            return light[:case["count"]]


# ---------------------------------------------------------------- prepare

def prepare(case, seed):
    rng = random.Random(seed)
    kind = case["kind"]
    if kind == "count":
        plan = tnc.plan_formula(_weighted(_formula(case), rng), heuristic=case["planner"], rank_cap=32)
        nb = tnc.workspace_bytes(plan, case["R"], case["path"], _primes(case))
        return {"kind": kind, "plan": plan, "R": case["R"], "path": case["path"], "primes": _primes(case),
                "ws": torch.empty(nb, dtype=torch.uint8, device="cuda")}
    if kind == "many":
        plans = tnc.plan_many([_weighted(f, rng) for f in _many_formulas(case)], heuristic="portfolio", rank_cap=32)
        nb = tnc.workspace_bytes_many(plans, case["R"], case["path"], len(plans))
        return {"kind": kind, "plans": plans, "R": case["R"], "path": case["path"],
                "ws": torch.empty(nb, dtype=torch.uint8, device="cuda")}
    if kind == "sliced":
        f = _weighted(I.cubic_vertex_cover(case["n"], case["graph"]), rng)
        plans, _ = tnc.plan_sliced(f, case["slices_log2"], heuristic="best", rank_cap=32)
        # room for every slice at once, so that they run merged
        nb = tnc.workspace_bytes_many(plans, case["R"], case["path"], len(plans)) + (1 << 16)
        return {"kind": kind, "plans": plans, "R": case["R"], "path": case["path"],
                "ws": torch.empty(nb, dtype=torch.uint8, device="cuda")}
    if kind == "batch":
        batch = tnc.Batch(_batch_plans(case, seed), n_residues=case["R"])
        ws = torch.empty(batch.workspace_bytes(), dtype=torch.uint8, device="cuda")
        batch.upload(ws)
        batch.launch(ws)
        return {"kind": kind, "batch": batch, "ws": ws, "upload": case["upload"], "out": batch.download_flat(ws)}
    x, t, params, m, v = _mlp_inputs(case, seed)
    rows = case["rows"]
    f32 = dict(dtype=torch.float32, device="cuda")
    if kind == "mlp_step":
        return {"kind": kind, "x": x, "t": t, "p0": params, "m0": m, "v0": v, "p": torch.empty_like(params),
                "m": torch.empty_like(m), "v": torch.empty_like(v), "g": torch.empty_like(params),
                "y": torch.empty(rows, **f32), "h1": torch.empty(rows, tnc.MLP_HIDDEN, **f32),
                "h2": torch.empty(rows, tnc.MLP_HIDDEN, **f32)}
    q = torch.empty(tnc.MLP_PARAMS, dtype=torch.bfloat16, device="cuda")
    tnc.mlp_to_bf16(params, q)
    return {"kind": kind, "x": x, "q": q, "y": torch.empty(rows, **f32)}


def _mlp_inputs(case, seed):
    """Rows of features of order 1 (about a quarter of them zero flags), regrets,
    and a scorer and its Adam state in mid-training."""
    g = torch.Generator().manual_seed(seed)
    rows, n = case["rows"], tnc.MLP_PARAMS
    x = torch.rand(rows, tnc.MLP_FEATURES, generator=g) * (torch.rand(rows, tnc.MLP_FEATURES, generator=g) > 0.25)
    t = torch.randn(rows, generator=g).abs() * 2
    f, h = tnc.MLP_FEATURES, tnc.MLP_HIDDEN
    he = [(f * h, (2 / f) ** 0.5), (h, 0.01), (h * h, (2 / h) ** 0.5), (h, 0.01), (h, (2 / h) ** 0.5), (1, 0.01)]
    params = torch.cat([std * torch.randn(size, generator=g) for size, std in he])
    m = 1e-3 * torch.randn(n, generator=g)
    v = 1e-6 * (0.5 + torch.rand(n, generator=g))
    return [a.float().cuda() for a in (x, t, params, m, v)]


# ---------------------------------------------------------------- run

STEP, LR = 100, 1e-3


def _results(counts):
    """Residues and exact values (128-byte little-endian integers) of counts."""
    return {"residues": np.concatenate([c.residues for c in counts]),
            "values": np.frombuffer(b"".join(v.to_bytes(128, "little") for c in counts for v in c.counts),
                                    dtype=np.uint8)}


def run(s):
    kind = s["kind"]
    if kind == "count":
        return _results([tnc.contract(s["plan"], s["R"], primes=s["primes"], workspace=s["ws"], path=s["path"])])
    if kind == "many":
        return _results(tnc.contract_many(s["plans"], s["R"], workspace=s["ws"], path=s["path"]))
    if kind == "sliced":
        return _results([tnc.contract_sliced(s["plans"], s["R"], workspace=s["ws"], path=s["path"])])
    if kind == "batch":
        if s["upload"]:
            s["batch"].upload(s["ws"])
        s["batch"].launch(s["ws"])
        residues, limbs, flags = s["batch"].download_flat(s["ws"], out=s["out"])
        return {"residues": residues, "limbs": limbs, "flags": flags}
    if kind == "mlp_step":
        for name in ("p", "m", "v"):
            s[name].copy_(s[name + "0"])
        tnc.mlp_forward(s["p"], s["x"], s["y"], s["h1"], s["h2"])
        tnc.mlp_backward(s["p"], s["x"], s["h1"], s["h2"], s["y"], s["t"], s["g"])
        tnc.mlp_adam(s["p"], s["g"], s["m"], s["v"], STEP, LR)
        return {"y": s["y"], "grads": s["g"], "params": s["p"], "m": s["m"], "v": s["v"]}
    tnc.mlp_forward_bf16(s["q"], s["x"], s["y"])
    return {"y": s["y"]}


# ---------------------------------------------------------------- work

def work(case):
    """Bytes: the formulas' weight tables (or the rows and parameters) read and
    the results written; flops: two per multiply-add of the plan, modular ones
    counted once per residue."""
    kind = case["kind"]
    if kind in ("mlp_step", "mlp_infer"):
        rows, n, h, f = case["rows"], tnc.MLP_PARAMS, tnc.MLP_HIDDEN, tnc.MLP_FEATURES
        fwd = 2.0 * rows * (f * h + h * h + h)
        if kind == "mlp_infer":
            return {"bytes": 4.0 * rows * (f + 1) + 2.0 * n, "flops": fwd}
        # x, t, parameters and Adam state in; y, gradients, parameters and Adam state out
        return {"bytes": 4.0 * rows * (f + 2) + 4.0 * 7 * n, "flops": 3.0 * fwd + 12.0 * n}
    if kind == "count":
        forms = [_formula(case)]
        plans = [tnc.plan_formula(forms[0], heuristic=case["planner"], rank_cap=32)]
    elif kind == "many":
        forms = _many_formulas(case)
        plans = tnc.plan_many(forms, heuristic="portfolio", rank_cap=32)
    elif kind == "sliced":
        forms = [I.cubic_vertex_cover(case["n"], case["graph"])]
        plans, _ = tnc.plan_sliced(forms[0], case["slices_log2"], heuristic="best", rank_cap=32)
    else:  # a sample of the batch, scaled
        sample = dict(case, count=min(case["count"], 128))
        forms, plans = _batch_formulas(case, 1, sample["count"]), _batch_plans(sample, 1)
    scale = case["count"] / len(forms) if kind == "batch" else 1.0
    read = sum(4.0 * sum(1 << len(vs) for vs in f.clauses) for f in forms)
    written = sum(8.0 * case["R"] * (1 << len(f.open_vars)) for f in forms)
    macs = sum(p.stats.total_macs for p in plans)
    return {"bytes": scale * (read + written), "flops": scale * 2.0 * macs * case["R"]}


# ---------------------------------------------------------------- exact

def exact(case, seed):
    """The scorer's outputs in 64 bits; counts are whole numbers and have no nearer value."""
    kind = case["kind"]
    if kind not in ("mlp_step", "mlp_infer"):
        return None
    h, f = tnc.MLP_HIDDEN, tnc.MLP_FEATURES
    x, t, params, m, v = _mlp_inputs(case, seed)
    if kind == "mlp_infer":
        params = params.to(torch.bfloat16)
    x, t, params, m, v = [a.double() for a in (x, t, params, m, v)]
    w1, b1, w2, b2, w3, b3 = torch.split(params, [f * h, h, h * h, h, h, 1])
    w1, w2 = w1.view(f, h), w2.view(h, h)
    h1 = torch.relu(x @ w1 + b1)
    h2 = torch.relu(h1 @ w2 + b2)
    y = h2 @ w3 + b3
    if kind == "mlp_infer":
        return {"y": y}
    dy = 2.0 * (y - t) / case["rows"]
    dh2 = dy[:, None] * w3 * (h2 > 0)
    dh1 = (dh2 @ w2.T) * (h1 > 0)
    grads = torch.cat([(x.T @ dh1).reshape(-1), dh1.sum(0), (h1.T @ dh2).reshape(-1), dh2.sum(0), h2.T @ dy,
                       dy.sum().reshape(1)])
    m = 0.9 * m + 0.1 * grads
    v = 0.999 * v + 0.001 * grads * grads
    params = params - LR * (m / (1 - 0.9 ** STEP)) / (torch.sqrt(v / (1 - 0.999 ** STEP)) + 1e-8)
    return {"y": y, "grads": grads, "params": params, "m": m, "v": v}
