"""The cases that performance work on this framework is measured by.

Every case is one call that a user's program makes through `binding.Context`:
a split search, a tree or forest or boosted ensemble trained from rows on the
GPU and read back, a forest's predictions, the proposal network's training.
Sizes are those of `workloads.SETTINGS` and of the tests, and odd ones beside
them. Inputs are drawn on the GPU with the distributions of `workloads`.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2208_07023_gb300 import binding as S

# Scores, splits and trees are fixed by the header's definition of every
# operation (sequential FP32 multiply-adds, exact integer histograms, one
# rounding per swarm operation), so another correct implementation differs
# only in the order of 64-bit sums (losses, means): a few units of 1e-16,
# and nothing in the 32-bit results.
SEARCH_TOL = {"rel": 1e-12, "max": 1e-10, "differ": 0.0}


def _tree(name, n, d, K, criterion, P, T, B, depth, min_leaf, levels, **more):
    c = dict(name=name, kind="tree", n=n, d=d, K=K, criterion=criterion, P=P, T=T, B=B,
             depth=depth, min_leaf=min_leaf, trees=1, proj="fp32", apso=False, top_n=0,
             levels=levels, mean_var=2.0)
    c.update(more)
    return c


def listed():
    return [
        # one node's swarm search: the smallest call, where launches and
        # latency count (an interactive split, a small subtree)
        dict(_tree("node_2000x16", 2000, 16, 2, "entropy", 32, 50, 64, 1, 1, 1.0), kind="node"),
        # a small ragged table, odd in every size: entropy trees on tabular data
        _tree("tree_7321x23_k7", 7321, 23, 7, "entropy", 37, 60, 100, 10, 5, 3.5),
        # adaptive PSO on a ragged table (the paper's accelerated swarm)
        _tree("apso_20011x33_k4", 20011, 33, 4, "gini", 40, 50, 128, 8, 20, 2.7, apso=True),
        # the ordinary classification tree
        _tree("tree_50000x64_k10", 50_000, 64, 10, "gini", 64, 100, 128, 8, 20, 4.2),
        # an ordinary regression tree of odd sizes, FP32 form
        _tree("regtree_30011x50", 30_011, 50, 0, "mse", 48, 60, 256, 10, 20, 9.0),
        # the large regression tree in the BF16 form with FP32 re-scoring
        _tree("regtree_200000x128_bf16", 200_000, 128, 0, "mse", 64, 80, 256, 10, 20, 10.0,
              proj="bf16"),
        # a bagged forest, every level of all trees one batch
        _tree("forest64_100000x32_k5", 100_000, 32, 5, "gini", 48, 60, 128, 8, 20, 2.9,
              trees=64),
        # SLR Boost: regression trees on residuals
        _tree("boost_200000x128", 200_000, 128, 0, "mse", 64, 40, 256, 6, 20, 6.0, kind="boost",
              rounds=2, lr=0.3),
        # SLM Boost: one regression tree per class and round, on classes that
        # overlap (on separable ones every tree is a stump)
        _tree("slmboost_50000x64_k10", 50_000, 64, 10, "mse", 64, 40, 128, 4, 20, 4.0,
              kind="boost", rounds=2, lr=0.5, mean_var=0.01),
        # a trained forest labels new rows
        _tree("predict64_100000x32_k5", 100_000, 32, 5, "gini", 48, 10, 128, 8, 20, 2.9,
              kind="predict", trees=64, train_n=20_000),
        # the proposal network learns from (statistics, best direction) pairs
        dict(name="proposal_train_1000", kind="proposal", n=1000, d=64, epochs=2, batch=64,
             lr=1e-3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["node", "tree", "tree", "regtree", "forest", "boost", "predict",
                       "proposal"])
    if kind == "proposal":
        return dict(kind="proposal", n=_log(rng, 60, 1500), d=rng.randint(4, 256), epochs=2,
                    batch=rng.choice([16, 32, 64, 128]), lr=1e-3)
    d = _log(rng, 4, 128)
    P, T, B = rng.randint(16, 64), rng.randint(20, 80), rng.choice([32, 64, 100, 128, 200, 256])
    K = rng.randint(2, 10)
    crit = rng.choice(["gini", "entropy"])
    min_leaf = rng.choice([1, 5, 20])
    if kind == "node":
        c = dict(_tree("", _log(rng, 500, 50_000), d, K, crit, P, T, B, 1, min_leaf, 1.0),
                 kind="node")
    elif kind == "tree":
        c = _tree("", _log(rng, 1000, 100_000), d, K, crit, P, T, B, rng.randint(3, 10), min_leaf,
                  3.0, apso=rng.random() < 0.2)
        if not c["apso"] and d >= 16 and rng.random() < 0.2:
            c["top_n"] = d // 2
    elif kind == "regtree":
        c = _tree("", _log(rng, 1000, 150_000), d, 0, "mse", P, T, B, rng.randint(3, 10), 20, 7.0,
                  proj=rng.choice(["fp32", "bf16"]))
    elif kind == "forest":
        trees = _log(rng, 2, 64)
        n = _log(rng, 1000, 100_000 if trees <= 16 else 40_000)
        c = _tree("", n, min(d, 64), K, crit, min(P, 48), min(T, 60), min(B, 128), 8, 20, 2.9,
                  trees=trees)
    elif kind == "predict":
        c = _tree("", _log(rng, 100, 200_000), min(d, 64), K, crit, 32, 10, 64, rng.randint(3, 10),
                  min_leaf, 2.9, kind="predict", trees=_log(rng, 1, 64), train_n=10_000)
    else:
        classes = rng.choice([0, K])
        n = _log(rng, 5000, 30_000) if classes else _log(rng, 1000, 100_000)
        c = _tree("", n, d, classes, "mse", P, min(T, 40), B, rng.randint(2, 6), 20, 5.0,
                  kind="boost", rounds=rng.randint(1, 3), lr=0.3, mean_var=0.64 / d)
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------

_CTX = {}


def _ctx():
    """A program's context: one for as long as it runs."""
    if "ctx" not in _CTX:
        _CTX["ctx"] = S.Context(0)
    return _CTX["ctx"]


def _mixture(g, n, d, K, mean_var, params=None):
    """workloads.gmm on the GPU: class means ~ N(0, mean_var I), one shared
    rotated covariance with eigenvalues log-uniform in [0.1, 10]."""
    dev = g.device
    if params is None:
        means = torch.randn(K, d, generator=g, device=dev) * math.sqrt(mean_var)
        q, r = torch.linalg.qr(torch.randn(d, d, generator=g, device=dev).cpu())
        q = (q * torch.sign(torch.diagonal(r))[None, :]).to(dev)
        lam = torch.exp(torch.rand(d, generator=g, device=dev) * math.log(100.0)) * 0.1
        params = (means, q, lam)
    means, q, lam = params
    labels = torch.randint(0, K, (n,), generator=g, device=dev, dtype=torch.int32)
    z = torch.randn(n, d, generator=g, device=dev)
    X = means[labels.long()] + (z * lam.sqrt()[None, :]) @ q.T
    return X.contiguous(), labels, params


def _halves(g, n, d):
    """workloads.single_node: two classes by the side of a random hyperplane,
    5 % of the labels flipped."""
    w = torch.randn(d, generator=g, device=g.device)
    X = torch.randn(n, d, generator=g, device=g.device)
    side = (X @ w >= 0).to(torch.int32)
    flip = torch.rand(n, generator=g, device=g.device) < 0.05
    return X.contiguous(), torch.where(flip, 1 - side, side).contiguous()


def _regression(g, n, d):
    """workloads.tanh_regression: eight tanh ridges and noise."""
    W = torch.randn(8, d, generator=g, device=g.device) / math.sqrt(d)
    X = torch.randn(n, d, generator=g, device=g.device)
    y = torch.tanh(X @ W.T).sum(1) + 0.1 * torch.randn(n, generator=g, device=g.device)
    return X.contiguous(), y.contiguous()


def _params(c, seed, criterion=None, T=None):
    trees = c["trees"]
    return S.make_params(criterion or c["criterion"], max(c["K"], 2), c["P"], T or c["T"], c["B"],
                         max_depth=c["depth"], min_leaf=c["min_leaf"], seed=seed, n_trees=trees,
                         bootstrap=trees > 1,
                         proj=S.SLM_PROJ_BF16_TOPK if c["proj"] == "bf16" else S.SLM_PROJ_FP32,
                         topk=8, apso=c["apso"], top_n=c["top_n"])


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda").manual_seed(seed)
    ctx = _ctx()
    st = {"case": c, "ctx": ctx}
    n, d = c["n"], c["d"]
    if c["kind"] == "proposal":
        # class statistics of d features and unit directions, zero past d
        stats = torch.zeros(n, S.PROP_K + 1, S.PROP_D, device="cuda")
        stats[:, :, :d] = torch.randn(n, S.PROP_K + 1, d, generator=g, device="cuda")
        stats[:, S.PROP_K, :d] = stats[:, S.PROP_K, :d] ** 2 + 0.1
        t = torch.zeros(n, S.PROP_D, device="cuda")
        t[:, :d] = stats[:, 0, :d] - stats[:, 1, :d]
        t = t / t.norm(dim=1, keepdim=True)
        st.update(stats=stats.reshape(n, S.PROP_IN).contiguous(), targets=t.contiguous(),
                  dims=torch.full((n,), d, dtype=torch.int32, device="cuda"),
                  prop=ctx.proposal(seed & 0x7FFFFFFF), seed=seed)
        return st
    st["params"] = _params(c, seed)
    if c["kind"] == "predict":
        Xt, lt, p = _mixture(g, c["train_n"], d, c["K"], c["mean_var"])
        st["forest"] = ctx.train_tree(st["params"], Xt, labels=lt)
        st["X"], _, _ = _mixture(g, n, d, c["K"], c["mean_var"], p)
    elif c["K"] == 0:
        st["X"], st["y"] = _regression(g, n, d)
    elif c["kind"] == "node" and c["K"] == 2:
        st["X"], st["labels"] = _halves(g, n, d)
    else:
        st["X"], st["labels"], _ = _mixture(g, n, d, c["K"], c["mean_var"])
    return st


# ---- one pass -----------------------------------------------------------------

def _stack(trees):
    return {k: np.stack([t[k] for t in trees]) for k in trees[0]}


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "proposal":
        losses = state["prop"].train(state["stats"], state["dims"], state["targets"],
                                     epochs=c["epochs"], batch=c["batch"], lr=c["lr"], seed=3)
        return dict(state["prop"].get(), losses=losses)
    p, X = state["params"], state["X"]
    y, labels = state.get("y"), state.get("labels")
    if c["kind"] == "node":
        r = ctx.node_split(p, X, labels=labels, y=y, node_uid=1, want_trace=True)
        return {k: r[k] for k in ("loss", "bin", "n_left", "n_right", "particle", "iter_of_best",
                                  "threshold", "norm", "direction", "gbest", "trace")}
    if c["kind"] == "predict":
        cls, val, _ = ctx.predict(state["forest"], X)
        return {"class": cls, "value": val}
    if c["kind"] == "boost":
        b = ctx.train_boost(p, X, y=y, labels=labels, n_rounds=c["rounds"],
                            learning_rate=c["lr"])
        k = max(c["K"], 1)
        out = _stack([b.tree(t).export() for t in range(c["rounds"] * k)])
        out["train_loss"] = b.train_loss
        return out
    f = ctx.train_tree(p, X, labels=labels, y=y)
    out = _stack([f.export(t) for t in range(c["trees"])])
    out["evaluations"] = f.info()["evaluations"]
    return out


# ---- what a pass cannot do without ------------------------------------------------

def work(case):
    c = case
    if c["kind"] == "proposal":
        # the inputs once, the weights in and out; forward and backward products
        w = S.PROP_IN * S.PROP_H + S.PROP_H * S.PROP_H + S.PROP_H * S.PROP_OUT
        steps = c["epochs"] * -(-c["n"] // c["batch"])
        return {"bytes": 4.0 * (c["n"] * (S.PROP_IN + S.PROP_D) + 2 * w * steps),
                "flops": 6.0 * w * c["n"] * c["epochs"]}
    n, d = c["n"], c["d"]
    if c["kind"] == "predict":
        # every row walks every tree (about 4 internal nodes each)
        return {"bytes": 4.0 * n * d + 12.0 * n, "flops": 2.0 * d * n * c["trees"] * 4}
    # every particle's projection of every searched node's rows: `levels` is
    # how often a row is searched on its way down (measured); bags hold
    # 1 - 1/e of the rows
    rows = n * c["trees"] * (0.632 if c["trees"] > 1 else 1.0) * min(c["levels"], c["depth"])
    if c["kind"] == "boost":
        rows *= c["rounds"] * max(c["K"], 1)
    dims = c["top_n"] or d
    return {"bytes": 4.0 * n * (d + 1), "flops": 2.0 * dims * rows * c["P"] * (c["T"] + 1)}


def tolerance(case):
    if case["kind"] == "proposal":
        # FP32 sums over up to 5,376 terms in another order, then Adam, whose
        # first steps take the sign of a gradient however small it is
        return {"rel": 2e-3, "max": 0.3}
    return dict(SEARCH_TOL)


def exact(case, seed):
    """None: a search's outputs are the path of a discrete search (one
    differently rounded score sends the swarm elsewhere), so 64 bits give
    another path; the network's weights follow the C++ library's shuffle."""
    return None
