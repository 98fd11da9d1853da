"""Workloads that stand for what a user has this library do, through its public entry points.

A case is a dict of plain values; prepare() makes its inputs on the GPU (or in
host memory where a program hands host buffers over), run() makes one call,
work() says what that call cannot do without.  Diagrams are the package's own
seeded synthetic ones: `uniform` (births uniform, exponential persistence, on a
1/256 grid), `lowerstar` (uint8 lower-star persistence of smoothed noise
images), `mixture` (continuous float32, few duplicates) and `gaussian`.

Returned are the values that the call defines: optimum, bounds, sizes, nodes,
network, gradients.  Left out are the counters of the path the solver took
(pivots, launches, times) and slack_quanta, the total flow of whichever of
several equally cheap flows it ended on.
"""
import itertools
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_2110_14734_gb300 import pdw1, synth

# pd_result fields that the inputs alone determine
RESULT = ("w1", "opt_quanta", "rwmd_quanta", "rwmd_A", "rwmd_B", "mass_A", "mass_B", "s", "coord_shift", "delta",
          "cell_quanta", "shift_quanta", "n_nodes", "n_arcs")

_GENERATE = {"uniform": synth.uniform_exp, "lowerstar": synth.lowerstar_u8, "mixture": synth.mixture_f32,
             "gaussian": synth.gaussian_pd}
_context = None


def listed():
    return [
        # one small pair, the latency of a single distance between two small diagrams (8-bit grid coordinates)
        {"name": "w1_uniform_2k", "path": "w1", "kind": "uniform", "n": 2000, "m": 2000, "eps": 0.1, "host": False},
        # one pair of the headline size, default options: 8-bit images' diagrams of 100,000 points
        {"name": "w1_lowerstar_100k", "path": "w1", "kind": "lowerstar", "n": 100000, "m": 100000, "eps": 0.05,
         "host": False},
        # the distance matrix of a set of small diagrams, as for a kernel or a clustering
        {"name": "batch_uniform_2k", "path": "batch", "kind": "uniform", "n": 2000, "count": 24, "eps": 0.1,
         "host": False},
        # the distance matrix of 18 headline-size diagrams handed over in host memory (153 pairs)
        {"name": "batch_lowerstar_100k", "path": "batch", "kind": "lowerstar", "n": 100000, "count": 18, "eps": 0.05,
         "host": True},
        # min-cost flow on a given sparse network (the empirical-complexity experiment's diagrams, s = 20)
        {"name": "mcf_gaussian_2k", "path": "mcf", "kind": "gaussian", "n": 2000, "m": 2000, "s": 20},
        # condensation of two large continuous diagrams onto a fine lattice
        {"name": "condense_mixture_1m", "path": "condense", "kind": "mixture", "n": 1000000, "m": 1000000,
         "cell": 200, "shift": 1},
        # lower bounds: a small pair (all latency; the filter in front of a solve) and a very large one
        {"name": "rwmd_uniform_2k", "path": "rwmd", "kind": "uniform", "n": 2000, "m": 2000},
        {"name": "rwmd_mixture_1m", "path": "rwmd", "kind": "mixture", "n": 1000000, "m": 1000000},
        # the sparse network itself, for a caller with a solver of its own
        {"name": "wspd_mixture_5k", "path": "wspd", "kind": "mixture", "n": 5000, "m": 5000, "s": 40, "tree": 0},
        # the size of the sparse network of the largest configuration
        {"name": "count_mixture_1m", "path": "count", "kind": "mixture", "n": 1000000, "m": 1000000, "eps": 0.1},
        # nearest diagram of a database of small diagrams
        {"name": "nn_uniform_96", "path": "nn", "kind": "uniform", "n": 700, "count": 96, "lo": 100, "hi": 2000,
         "eps": 0.05},
        # one training step's loss and gradients of the warm-start network (2,048 rows a step)
        {"name": "ws_grad_2k", "path": "ws", "rows": 2048, "op": "grad"},
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["w1", "w1", "batch", "batch", "mcf", "condense", "rwmd", "wspd", "count", "nn", "ws"])
    if path == "w1":
        kind = rng.choice(["uniform", "lowerstar", "mixture"])
        lo, hi = {"uniform": (200, 2500), "lowerstar": (1000, 100000), "mixture": (200, 2000)}[kind]
        eps = {"uniform": (0.1, 0.05), "lowerstar": (0.05, 0.01), "mixture": (0.1,)}[kind]
        return {"path": path, "kind": kind, "n": _size(rng, lo, hi), "m": _size(rng, lo, hi), "eps": rng.choice(eps),
                "host": rng.random() < 0.3}
    if path == "batch":
        kind = rng.choice(["uniform", "lowerstar"])
        lo, hi = {"uniform": (200, 2000), "lowerstar": (2000, 60000)}[kind]
        return {"path": path, "kind": kind, "n": _size(rng, lo, hi), "count": rng.randint(3, 20),
                "eps": 0.1 if kind == "uniform" else 0.05, "host": rng.random() < 0.5}
    if path == "mcf":
        return {"path": path, "kind": "gaussian", "n": _size(rng, 200, 2000), "m": _size(rng, 200, 2000),
                "s": rng.choice([8, 10, 16, 20])}
    if path == "condense":
        kind, cell = rng.choice(["mixture", "uniform", "lowerstar"]), _size(rng, 1, 6000)
        hi = 100000 if kind == "lowerstar" else 1000000
        return {"path": path, "kind": kind, "n": _size(rng, 1000, hi), "m": _size(rng, 1000, hi), "cell": cell,
                "shift": cell // 200}
    if path == "rwmd":
        kind = rng.choice(["mixture", "uniform", "lowerstar"])
        hi = 100000 if kind == "lowerstar" else 1000000
        return {"path": path, "kind": kind, "n": _size(rng, 1000, hi), "m": _size(rng, 1000, hi)}
    if path == "wspd":
        return {"path": path, "kind": rng.choice(["mixture", "gaussian"]), "n": _size(rng, 200, 5000),
                "m": _size(rng, 200, 5000), "s": rng.choice([8, 20, 40]), "tree": rng.randint(0, 1)}
    if path == "count":
        return {"path": path, "kind": "mixture", "n": _size(rng, 5000, 500000), "m": _size(rng, 5000, 500000),
                "eps": rng.choice([0.1, 0.2])}
    if path == "nn":
        return {"path": path, "kind": "uniform", "n": _size(rng, 100, 1000), "count": _size(rng, 12, 96), "lo": 100,
                "hi": _size(rng, 500, 2000), "eps": rng.choice([0.1, 0.05])}
    return {"path": path, "rows": _size(rng, 100, 20000), "op": rng.choice(["forward", "grad"])}


def _shared():
    """The context that a program keeps for all its calls."""
    global _context
    if _context is None:
        _context = pdw1.pd_create(0)
    return _context


def _diagrams(case, seed, sizes, host=False):
    """One diagram per size; generating is host work, spread over a few threads."""
    make = _GENERATE[case["kind"]]
    with ThreadPoolExecutor(12) as pool:
        got = list(pool.map(lambda t: make(t[1], 1000 * (seed % 1000003) + t[0]), enumerate(sizes)))
    return [torch.from_numpy(x).pin_memory() if host else torch.from_numpy(x).cuda() for x in got]


def _ws_arrays(case, seed):
    rng = np.random.default_rng(seed)
    rows = case["rows"]
    params = rng.standard_normal(pdw1.WS_NPARAMS) * 0.1
    feats = rng.standard_normal((rows, pdw1.WS_NFEAT))
    # the values that the entry points keep: parameters in float32, features in bf16
    params = params.astype(np.float32)
    feats = torch.from_numpy(feats).bfloat16().float().numpy()
    target = (0.3 * rng.standard_normal(rows)).astype(np.float32)
    mask = (rng.random(rows) < 0.9).astype(np.float32)
    return params, feats, target, mask


def _padded(sizes):
    """Output arrays of a size that the case alone gives: the values, then -1."""
    return {k: torch.full((n,), -1, dtype=torch.int32 if k in ("X", "Y", "head") else torch.int64, device="cuda")
            for k, n in sizes.items()}


def _into(out, got):
    for k, t in out.items():
        t[: got[k].numel()].copy_(got[k])
    return out


def prepare(case, seed):
    path = case["path"]
    if path == "batch":
        ds = _diagrams(case, seed, [case["n"]] * case["count"], case["host"])
        pairs = list(itertools.combinations(range(case["count"]), 2))
        return dict(case=case, ctx=_shared(), A=[ds[i] for i, _ in pairs], B=[ds[j] for _, j in pairs])
    if path == "nn":
        sizes = synth.db_sizes(case["count"], seed % 1000003, case["lo"], case["hi"])
        ds = _diagrams(case, seed, [case["n"]] + [int(k) for k in sizes])
        ctx = pdw1.pd_create(0)  # a database lives in its context
        pdw1.pd_db_build(ctx, ds[1:])
        return dict(case=case, ctx=ctx, query=ds[0])
    if path == "ws":
        params, feats, target, mask = _ws_arrays(case, seed)
        ctx = pdw1.pd_create(0)  # the network lives in its context
        pdw1.pd_ws_set_params(ctx, params)
        return dict(case=case, ctx=ctx, feats=feats, target=target, mask=mask)
    A, B = _diagrams(case, seed, [case["n"], case["m"]], case.get("host", False))
    state = dict(case=case, ctx=_shared(), A=A, B=B)
    n = case["n"] + case["m"]
    if path == "condense":
        state["out"] = _padded({k: n for k in ("X", "Y", "cntA", "cntB", "morton")})
    if path == "wspd":  # at most 50 s arcs a node, a bound for these diagrams
        arcs = n * min(n, 50 * case["s"]) + 2 * n + 1
        state["net_out"] = _padded({"row_ptr": n + 3, "head": arcs, "cost": arcs, "supply": n + 2})
        state["nodes_out"] = _padded({k: n for k in ("X", "Y", "cntA", "cntB")})
    if path in ("wspd", "mcf"):
        state["nodes"] = pdw1.pd_condense(state["ctx"], A, B, 1, 0)
    if path == "mcf":
        state["net"] = pdw1.pd_wspd_sparsify(state["ctx"], state["nodes"], case["s"])
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    path = case["path"]
    if path == "w1":
        r = pdw1.pd_w1_approx(ctx, state["A"], state["B"], case["eps"])
        return {k: r[k] for k in RESULT}
    if path == "batch":
        rows = pdw1.pd_w1_approx_batch(ctx, state["A"], state["B"], case["eps"])
        return {k: np.array([r[k] for r in rows]) for k in RESULT}
    if path == "mcf":
        return pdw1.pd_mcf_solve(ctx, state["net"])[0]
    if path == "condense":
        nodes = pdw1.pd_condense(ctx, state["A"], state["B"], case["cell"], case["shift"])
        return {"n_nodes": nodes["n_nodes"], "nodes": _into(state["out"], nodes)}
    if path == "rwmd":
        return pdw1.pd_rwmd_lower_bound(ctx, state["A"], state["B"])
    if path == "wspd":
        net, nodes = pdw1.pd_wspd_sparsify_tree(ctx, state["nodes"], case["s"], case["tree"])
        return {"n_nodes": net["n_nodes"], "n_arcs": net["n_arcs"], "net": _into(state["net_out"], net),
                "nodes": _into(state["nodes_out"], nodes)}
    if path == "count":
        r = pdw1.pd_w1_sparsify_count(ctx, state["A"], state["B"], case["eps"])
        return {k: r[k] for k in RESULT if k not in ("w1", "opt_quanta")}
    if path == "nn":
        r = pdw1.pd_nn_search(ctx, state["query"], case["eps"])
        return {"nn_index": r["nn_index"], "nn_opt_quanta": r["nn_opt_quanta"], "nn_w1": r["nn_w1"],
                "opt": np.array(r["opt"]), "lb": np.array(r["lb"]), "wcd": np.array(r["wcd"])}
    if case["op"] == "forward":
        return pdw1.pd_ws_forward(ctx, state["feats"])
    loss, grad = pdw1.pd_ws_grad(ctx, state["feats"], state["target"], state["mask"])
    return {"loss": loss, "grad": grad}


def work(case):
    """Inputs read once and outputs written once; the exact optimum has no smaller certain floor."""
    path = case["path"]
    if path == "ws":
        macs = 72 * 128 + 128 * 128 + 128
        nbytes = case["rows"] * 4 * 72 + 4 * pdw1.WS_NPARAMS
        if case["op"] == "forward":
            return {"bytes": nbytes + 4 * case["rows"], "flops": 2 * macs * case["rows"]}
        return {"bytes": nbytes + 8 * case["rows"] + 4 * pdw1.WS_NPARAMS, "flops": 6 * macs * case["rows"]}
    point = 2 if case["kind"] == "lowerstar" else 8
    if path == "batch":
        return {"bytes": point * case["n"] * case["count"] + 8 * len(RESULT) * case["count"] * (case["count"] - 1) // 2,
                "flops": 0}
    if path == "nn":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        return {"bytes": int(point * (case["n"] + mean * case["count"]) + 24 * case["count"]), "flops": 0}
    n = case["n"] + case["m"]
    if path == "condense":  # out: X, Y int32, two int64 counts, an int64 code per node (a uint8 grid has few nodes)
        nodes = min(n, 33000) if case["kind"] != "mixture" else n
        return {"bytes": point * n + 32 * nodes, "flops": 0}
    if path in ("wspd", "mcf"):  # arcs: head and cost, 12 bytes each; about 12 s (mixture), 25 s (gaussian) a node
        arcs = n * min(n, (12 if case["kind"] == "mixture" else 25) * case["s"])
        return {"bytes": 32 * n + 12 * arcs, "flops": 0}
    return {"bytes": point * n + 8 * len(RESULT), "flops": 0}


def exact(case, seed):
    """The warm-start network in 64 bits; the other outputs are whole numbers, or a whole number times 2^-k."""
    if case["path"] != "ws":
        return None
    params, feats, target, mask = (torch.from_numpy(x).double() for x in _ws_arrays(case, seed))
    cut = [72 * 128, 128, 128 * 128, 128, 128, 1]
    w1, b1, w2, b2, w3, b3 = torch.split(params, cut)
    # weights are kept in bf16, biases in float32
    w1, w2, w3 = (w.float().bfloat16().double() for w in (w1, w2, w3))
    leaves = [w.clone().requires_grad_(True) for w in (w1, b1, w2, b2, w3, b3)]
    w1, b1, w2, b2, w3, b3 = leaves
    h = torch.relu(feats @ w1.view(72, 128) + b1)
    h = torch.relu(h @ w2.view(128, 128) + b2)
    y = h @ w3 + b3
    if case["op"] == "forward":
        return y.detach().numpy()
    loss = (mask * (y - target) ** 2).sum() / case["rows"]
    loss.backward()
    return {"loss": float(loss), "grad": torch.cat([w.grad for w in leaves]).numpy()}
