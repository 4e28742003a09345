"""The work that users of the community-based ADMM GCN trainer have it do, as cases that can be timed and compared.

``listed()`` names the cases, ``draw`` gives more of the same ranges, ``prepare`` makes what a program has in
hand before the call (seeded synthetic inputs and, where such a program keeps one, the handle), ``run`` is one
pass through the public entry points of ``paper_2112_09335_b200.binding.GcnAdmm``.  A case is a dict of plain
values:

  path       what the program does (see ``run``): "fit", "resume", "train", "curve", "predict", "propagate" or
             "propagate_static"
  n, edges   nodes and undirected edges of the graph;  alpha: Pareto tail of the node weights (0 = equal weights)
  blocks     planted blocks (also the label structure);  comm: communities of the trainer
  widths     "C_0-C_1-..-C_L";  feat: how the node features are distributed;  train: share of the nodes in training
  passes     passes of Algorithm 1 in one run;  schedule, dual_mode: the trainer's options of those names
  width      columns of the propagated matrix ("propagate" paths)

The graphs follow the recipe of ``paper_2112_09335_b200/inputs.py`` (a degree-corrected block model, 85 % of the
draws inside a block, ids shuffled), drawn on the GPU so that the largest one takes a fraction of a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2112_09335_b200 import binding

WARM_PASSES = 3     # passes a kept handle has behind it: every block of the trainer is moving by then


def listed():
    return [
        # The smallest call: one propagation in a loop that may not allocate, on a small citation graph.
        dict(name="propagate_static small", path="propagate_static", n=2708, edges=5300, alpha=1.5, blocks=7, comm=8, width=16),
        # A preemptible job on a toy block model: load a checkpoint, ten passes, save it.  Launch latency is all there is.
        dict(name="resume tiny-sbm", path="resume", n=1000, edges=4500, alpha=0.0, blocks=4, comm=4, widths="128-16-7",
             feat="bow", train=0.14, passes=10, schedule=0, dual_mode=0),
        # A whole small experiment from host arrays: create, 20 passes, weights and predictions (wide bag-of-words features).
        dict(name="fit citation-small", path="fit", n=2708, edges=5300, alpha=1.5, blocks=7, comm=8, widths="1433-16-7",
             feat="bow", train=0.052, passes=20, schedule=0, dual_mode=0),
        # The same kind of graph seven times larger, few classes, textbook dual update, resumed from a checkpoint.
        dict(name="resume citation-medium", path="resume", n=19717, edges=44300, alpha=1.5, blocks=3, comm=16, widths="500-128-3",
             feat="tfidf", train=0.003, passes=6, schedule=0, dual_mode=1),
        # The paper's convergence curve (1000 hidden units, 3 communities): the objective and accuracy after every pass.
        dict(name="curve table2-shaped", path="curve", n=13752, edges=206280, alpha=1.5, blocks=10, comm=3, widths="767-1000-10",
             feat="bow", train=0.073, passes=2, schedule=0, dual_mode=0),
        # The serial schedule the paper compares with, on ragged sizes (no width a multiple of four, odd communities).
        dict(name="train serial ragged", path="train", n=30011, edges=240077, alpha=1.3, blocks=23, comm=13, widths="301-137-61-23",
             feat="normal", train=0.3, passes=3, schedule=1, dual_mode=0),
        # Training in progress on a large graph: a few passes, then weights, step sizes and objective are looked at.
        dict(name="train powerlaw-large", path="train", n=169343, edges=1170000, alpha=1.1, blocks=40, comm=32,
             widths="128-256-256-40", feat="normal", train=0.54, passes=3, schedule=0, dual_mode=0),
        # The same workload as one program run from host arrays.
        dict(name="fit powerlaw-large", path="fit", n=169343, edges=1170000, alpha=1.1, blocks=40, comm=32,
             widths="128-256-256-40", feat="normal", train=0.54, passes=8, schedule=0, dual_mode=0),
        # Inference with trained weights over all nodes: logits and labels on the host.
        dict(name="predict powerlaw-large", path="predict", n=169343, edges=1170000, alpha=1.1, blocks=40, comm=32,
             widths="128-256-256-40", feat="normal", train=0.54, schedule=0, dual_mode=0),
        # Feature smoothing A~ X between device buffers.
        dict(name="propagate powerlaw-large", path="propagate", n=169343, edges=1170000, alpha=1.1, blocks=40, comm=32, width=128),
        # The largest workload of the benchmark: two passes of a training run, then weights, step sizes and objective.
        dict(name="train powerlaw-xlarge", path="train", n=2449029, edges=61900000, alpha=1.0, blocks=47, comm=64,
             widths="100-256-256-47", feat="normal", train=0.08, passes=2, schedule=0, dual_mode=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    path = rng.choice(["resume", "fit", "train", "train", "curve", "predict", "propagate", "propagate_static"])
    lo, hi = dict(resume=(1000, 30000), fit=(1000, 200000), train=(20000, 2400000), curve=(2000, 60000), predict=(2000, 1000000),
                  propagate=(5000, 1000000), propagate_static=(1000, 40000))[path]
    n = _log_int(rng, lo, hi) | 1
    deg = math.exp(rng.uniform(math.log(4.0), math.log(50.0)))
    blocks = rng.randint(3, 47)
    comm = blocks if rng.random() < 0.3 else rng.randint(2, 64)
    case = dict(path=path, n=n, edges=int(n * deg / 2), alpha=rng.choice([0.0, 1.0, 1.1, 1.3, 1.5]), blocks=blocks, comm=comm)
    if path.startswith("propagate"):
        top = 256 if path == "propagate" else min(256, (4 << 20) // n - 3)
        case["width"] = _log_int(rng, 3, max(4, top))
        return case
    layers = rng.choice([2, 2, 3])
    hidden = [_log_int(rng, 16, 1000 if n < 20000 and layers == 2 else 256) for _ in range(layers - 1)]
    c0 = _log_int(rng, 100, 1433 if n < 20000 else 300)
    feat = rng.choice(["normal", "bow", "tfidf"])
    case.update(widths="-".join(str(w) for w in [c0, *hidden, blocks]), feat=feat, train=round(math.exp(rng.uniform(math.log(0.01), math.log(0.6))), 4),
                schedule=0, dual_mode=0)
    if path != "predict":
        case["passes"] = dict(resume=rng.randint(3, 6), fit=rng.randint(4, 8), train=2, curve=2)[path]
        case["schedule"] = 1 if rng.random() < 0.2 else 0
        case["dual_mode"] = 1 if rng.random() < 0.3 else 0
    return case


def draw(rng):
    """One more case of the ranges of ``listed`` that asks for at most half of the largest listed one's bytes and flops."""
    top = work(listed()[-1])
    while True:
        case = _draw_once(rng)
        w = work(case)
        if w["bytes"] <= 0.5 * top["bytes"] and w["flops"] <= 0.5 * top["flops"]:
            return case


# ---- inputs ----------------------------------------------------------------------------------------

def _widths(case):
    return [int(w) for w in case["widths"].split("-")]


def _graph(case, gen):
    """(row_ptr int64, col_idx int32, block int64, community int32) on the GPU; block and community per shuffled id."""
    n, edges, blocks, alpha = case["n"], case["edges"], case["blocks"], case["alpha"]
    ids = torch.arange(n, device="cuda")
    block = ids * blocks // n                      # contiguous before the shuffle
    w = torch.ones(n, dtype=torch.float64, device="cuda")
    if alpha > 0:
        w = (1.0 - torch.rand(n, generator=gen, dtype=torch.float64, device="cuda")) ** (-1.0 / alpha)
        cap = math.sqrt(n * 2.0 * edges / n)
        for _ in range(3):                         # no expected degree above sqrt(n * mean degree)
            w = torch.minimum(w, cap * w.mean() * n / (2.0 * edges))
    # whole-number weights: their running sums are exact, so the same seed gives the same graph
    wi = torch.clamp((w * (2.0 ** 20)).to(torch.int64), min=1)
    cdf = torch.cumsum(wi, 0)
    total = int(cdf[-1])
    draws = int(edges * 1.1)

    def pick(lo, hi):                              # node ~ weight among those whose running sum lies in [lo, hi)
        at = (torch.rand(draws, generator=gen, dtype=torch.float64, device="cuda") * (hi - lo)).to(torch.int64) + lo
        return torch.clamp(torch.searchsorted(cdf, at, right=True), max=n - 1)

    u = pick(0, total)
    ends = torch.searchsorted(block, torch.arange(blocks, device="cuda"), right=True)
    hi = cdf[ends - 1]
    lo = torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), hi[:-1]])
    intra = torch.rand(draws, generator=gen, device="cuda") < 0.85
    bu = block[u]
    v = pick(torch.where(intra, lo[bu], 0), torch.where(intra, hi[bu], total))
    del bu, intra
    relabel = torch.randperm(n, generator=gen, device="cuda")
    u, v = relabel[u], relabel[v]
    key = torch.minimum(u, v) * n + torch.maximum(u, v)
    key = torch.unique(key[u != v])
    u, v = key // n, key % n
    key = torch.sort(torch.cat([key, v * n + u]))[0]
    col_idx = (key % n).to(torch.int32)
    row_ptr = torch.searchsorted(key, torch.arange(n + 1, device="cuda") * n)
    shuffled_block, community = torch.empty_like(block), torch.empty(n, dtype=torch.int32, device="cuda")
    shuffled_block[relabel] = block
    community[relabel] = (ids * case["comm"] // n).to(torch.int32)
    return row_ptr, col_idx, shuffled_block, community


def _features(case, c0, y, gen):
    n, classes = case["n"], case["blocks"]
    if case["feat"] == "normal":
        return torch.randn(n, c0, generator=gen, device="cuda")
    draws = torch.rand(n, c0, generator=gen, device="cuda")
    if case["feat"] == "bow":                      # words, three times as likely in the columns of the node's class
        p = min(0.3, 20.0 / c0)
        own = y[:, None] == (torch.arange(c0, device="cuda") * classes // c0)[None, :]
        return (draws < torch.where(own, 3.0 * p, p)).float()
    x = torch.randn(n, c0, generator=gen, device="cuda").abs() * (draws < 0.1)
    x[torch.arange(n, device="cuda"), torch.randint(0, c0, (n,), generator=gen, device="cuda")] += 0.5   # no empty row
    return x / x.norm(dim=1, keepdim=True)


def _problem(case, seed):
    """The inputs of Algorithm 1 as device tensors, and the initial weights as host arrays."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    row_ptr, col_idx, block, community = _graph(case, gen)
    widths = _widths(case) if "widths" in case else [4, 4, case["blocks"]]   # propagation only: the network is not used
    if "widths" in case:
        X = _features(case, widths[0], block, gen)
        mask = torch.rand(case["n"], generator=gen, device="cuda") < case["train"]
    else:
        X = torch.zeros(case["n"], widths[0], device="cuda")
        mask = torch.zeros(case["n"], dtype=torch.bool, device="cuda")
    rng = np.random.default_rng(seed)
    glorot = [(rng.uniform(-1.0, 1.0, (a, b)) * math.sqrt(6.0 / (a + b))).astype(np.float32) for a, b in zip(widths, widths[1:])]
    return dict(row_ptr=row_ptr, col_idx=col_idx, X=X, y=block.to(torch.int32), mask=mask.to(torch.uint8), community=community), widths, glorot


def _create(case, arrays, widths, weights, stream):
    """A handle from host arrays or device tensors."""
    a = {k: v.data_ptr() if isinstance(v, torch.Tensor) else v for k, v in arrays.items()}
    return binding.GcnAdmm(case["n"], a["row_ptr"], a["col_idx"], a["X"], a["y"], a["mask"], widths, case["comm"], a["community"], weights,
                           schedule=case.get("schedule", 0), dual_mode=case.get("dual_mode", 0), stream=stream.cuda_stream)


def _save(g):
    """A checkpoint: the whole state of the trainer as host arrays."""
    ck = {"U": g.get_state(binding.ST_U)}
    for l in range(1, g.L + 1):
        ck["W%d" % l] = g.get_state(binding.ST_W, l)
        ck["Z%d" % l] = g.get_state(binding.ST_Z, l)
        ck["tau%d" % l] = g.get_state(binding.ST_TAU, l)
        if l < g.L:
            ck["theta%d" % l] = g.get_state(binding.ST_THETA, l)
    return ck


def _look(g):
    """What a training loop looks at between passes: weights, step sizes, objective and accuracy."""
    return {"W": [g.weights(l) for l in range(1, g.L + 1)], "tau": [g.get_state(binding.ST_TAU, l) for l in range(1, g.L + 1)],
            "theta": [g.get_state(binding.ST_THETA, l) for l in range(1, g.L)], "objective": g.objective()}


def _load(g, ck):
    g.set_state(binding.ST_U, 0, ck["U"])
    for l in range(1, g.L + 1):
        g.set_state(binding.ST_W, l, ck["W%d" % l])
        g.set_state(binding.ST_Z, l, ck["Z%d" % l])
        g.set_state(binding.ST_TAU, l, ck["tau%d" % l])
        if l < g.L:
            g.set_state(binding.ST_THETA, l, ck["theta%d" % l])


def prepare(case, seed):
    arrays, widths, weights = _problem(case, seed)
    path = case["path"]
    # training and inference work on a stream of their own, a propagation in the middle of a torch program on the current one
    stream = torch.cuda.current_stream() if path.startswith("propagate") else torch.cuda.Stream()
    torch.cuda.synchronize()
    state = dict(case=case, widths=widths, weights=weights, stream=stream)
    if path == "fit":
        state["arrays"] = {k: v.cpu().numpy() for k, v in arrays.items()}
        return state
    g = state["g"] = _create(case, arrays, widths, weights, stream)
    if path.startswith("propagate"):
        gen = torch.Generator(device="cuda").manual_seed(seed + 1)
        state["x"] = torch.randn(case["n"], case["width"], generator=gen, device="cuda")
        state["out"] = torch.empty_like(state["x"])
        return state
    g.step(WARM_PASSES)
    if path == "resume":
        state["checkpoint"] = _save(g)
    return state


# ---- one pass --------------------------------------------------------------------------------------

def run(state):
    case, g = state["case"], state.get("g")
    path = case["path"]
    if path == "propagate":
        g.propagate(state["x"].data_ptr(), case["width"], state["out"].data_ptr())
        return state["out"]
    if path == "propagate_static":
        g.propagate_static(state["x"].data_ptr(), case["width"], state["out"].data_ptr())
        return state["out"]
    if path == "predict":
        return g.predict()
    if path == "curve":                            # the objective's parts and the accuracy after every pass, then the weights
        curve = []
        for _ in range(case["passes"]):
            g.step(1)
            curve.append(g.objective())
        return {"curve": np.stack(curve), "W": [g.weights(l) for l in range(1, g.L + 1)]}
    if path == "resume":
        _load(g, state["checkpoint"])
        g.step(case["passes"])
        return _save(g)
    if path == "fit":
        g = _create(case, state["arrays"], state["widths"], state["weights"], state["stream"])
        g.step(case["passes"])
        logits, labels = g.predict()
        out = {"W": [g.weights(l) for l in range(1, g.L + 1)], "logits": logits, "labels": labels}
        g.destroy()
        return out
    g.step(case["passes"])
    return _look(g)


# ---- what a pass cannot do without -----------------------------------------------------------------

def work(case):
    """Bytes and fp32 operations of one ``run``: per pass of Algorithm 1 the graph and P_1 read once, the state read and
    written once; the products and sparse products of the method."""
    n, nnz = case["n"], 2 * case["edges"] + case["n"]
    graph = 4.0 * nnz + 8.0 * n                    # column ids, row pointers and normaliser
    if "width" in case:
        return {"bytes": graph + 8.0 * n * case["width"], "flops": 2.0 * nnz * case["width"]}
    c = _widths(case)
    L = len(c) - 1
    dense = sum(c[l - 1] * c[l] for l in range(1, L + 1))
    forward = 2.0 * n * dense + 2.0 * nnz * sum(c[1:L])
    if case["path"] == "predict":
        return {"bytes": graph + 4.0 * n * (c[0] + c[L] + 1) + 4.0 * dense, "flops": forward}
    state = n * (sum(c[1:]) + c[L]) + dense        # Z_1..Z_L, U, W
    flops = 0.0
    for l in range(1, L + 1):
        flops += 2.0 * n * c[l - 1] * c[l] * (2 if l == 1 else 3)             # P^T R and P grad; P W where P has moved
        if l < L:
            flops += 4.0 * n * c[l] * c[l + 1] + 2.0 * nnz * (2 * c[l + 1] + c[l])   # gradient, its image; A~ R', A~ T, A~ Z
    one = {"bytes": graph + 4.0 * n * c[0] + 8.0 * state, "flops": flops}
    total = {k: v * case["passes"] for k, v in one.items()}
    looks = dict(curve=case["passes"], train=1).get(case["path"], 0)   # objectives asked for
    total["flops"] += looks * forward
    total["bytes"] += looks * (graph + 4.0 * n * c[0] + 4.0 * state)
    if case["path"] == "resume":
        total["bytes"] += 8.0 * state              # checkpoint in and out
    if case["path"] == "fit":
        total["bytes"] += graph + 4.0 * n * (c[0] + c[L] + 1)              # the inputs themselves; logits and labels
        total["flops"] += forward
    return total


def tolerance(case):
    """fp32 throughout.  A propagation or a forward pass is off by sums of fp32 roundings.  The passes of Algorithm 1 work on
    differences of nearly equal fp32 numbers (Z_l - f(H_l)) and on step sizes decided from their sums, so they amplify roundings from
    pass to pass: two fp32 forms of the products (fused multiply-adds, and split TF32 on the tensor cores) end a run 1e-7 (small) to
    5e-4 (large) of the state's norm apart.  The runs are kept short for that reason."""
    if "width" in case:
        return {"rel": 1e-6, "max": 1e-5}
    if case["path"] == "predict":
        return {"rel": 3e-4, "max": 3e-2, "differ": 1e-3}
    return {"rel": 2e-4, "max": 1e-2, "differ": 1e-3} if case["n"] < 5000 else {"rel": 2e-3, "max": 0.1, "differ": 1e-3}
