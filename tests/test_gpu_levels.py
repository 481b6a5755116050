"""The per-level tree kernels (statistics, sides, decisions, scatter, gather)
at the widths where their row copies and products change form: rows of whole
16-byte words and not, up to and beyond the 256 words that a block copies at a time, and the
32-feature turns of the side's product with and without a remainder; nodes of
one and several 256-row tiles, more than 64 of them (the per-node kernels'
fetches). Trees equal the oracle's."""
import numpy as np
import pytest

import oracle as O
from paper_2208_07023_gb300 import workloads as W
from tests.gpu_util import context, gpu_params, oracle_params
from tests.test_gpu_parity import _check_tree_up_to_near_ties, _compare_tree

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = context()
    yield c
    c.close()


@pytest.mark.parametrize("crit,n,d", [
    ("gini", 17000, 1), ("gini", 2000, 4), ("gini", 700, 31), ("gini", 700, 36),
    ("gini", 600, 261), ("gini", 513, 1024),
    ("mse", 17000, 2), ("mse", 8300, 32), ("mse", 255, 257),
])
def test_tree_matches_oracle(ctx, crit, n, d):
    from paper_2208_07023_gb300 import binding as S
    K, B = (5, 32) if crit == "gini" else (0, 32)
    wl = W.gmm(n, d, K, seed=d) if K else W.tanh_regression(n, d, seed=d)
    lab, y = (wl.labels, None) if K else (None, wl.y)
    gp = gpu_params(S, crit, K, 16, 3, B, min_leaf=5, max_depth=3, seed=4)
    op = oracle_params(O, crit, K, 16, 3, B, min_leaf=5, max_depth=3, seed=4)
    g = ctx.train_tree(gp, wl.X, labels=lab, y=y).export(0)
    r = O.train_tree(op, wl.X, lab, y)
    assert (r.kind == 1).any()
    if K:
        inner, present = _compare_tree(g, r, d)
        assert np.array_equal(g["loss"][inner], r.loss[inner])
        assert np.array_equal(g["leaf_class"][present], r.leaf_class[present])
    elif _check_tree_up_to_near_ties(g, r, op, wl.X, None, wl.y) == 0:
        present = r.kind >= 0
        assert np.allclose(g["leaf_value"][present], r.leaf_value[present], rtol=1e-12, atol=1e-12)


@pytest.mark.parametrize("d,trees", [(5, 1), (8, 1), (54, 1), (16, 9), (260, 2), (452, 1),
                                     (452, 3), (601, 1), (900, 1)])
def test_prediction_does_not_depend_on_the_tile(ctx, d, trees):
    """Tiles of 32 to 256 rows (fewer rows a block where there are few),
    staged by 4- or 16-byte copies, or (one tree in long batches from 192
    features, or 425 whose rows are not whole 16-byte words; 900 features) read
    where they are: every row's class and leaves."""
    from paper_2208_07023_gb300 import binding as S
    wl = W.gmm(40000, d, 4, seed=d)
    p = gpu_params(S, "gini", 4, 16, 3, 32, min_leaf=5, max_depth=5, seed=6, n_trees=trees,
                   bootstrap=trees > 1)
    f = ctx.train_tree(p, wl.X[:3000], labels=wl.labels[:3000])
    cls, _, leaf = ctx.predict(f, wl.X, want_leaf=True)
    for n in (1, 31, 33, 4833, 19457, 38913):
        c, _, lf = ctx.predict(f, wl.X[:n], want_leaf=True)
        assert np.array_equal(c, cls[:n]) and np.array_equal(lf, leaf[:n]), n
    f.free()


@pytest.mark.parametrize("n,d", [(1, 1024), (3, 8), (5, 130), (9, 1001), (17, 1000), (63, 36),
                                 (255, 1024), (257, 33), (1300, 60), (77903, 3)])
def test_gather_of_few_and_many_rows(ctx, n, d):
    """4 to 256 entries a block: a subset's scores are the oracle's."""
    from paper_2208_07023_gb300 import binding as S
    wl = W.gmm(max(2 * n, 64), d, 4, seed=d)
    rng = np.random.default_rng(n)
    idx = rng.choice(len(wl.X), n, replace=False).astype(np.int32)
    pos = rng.uniform(-1, 1, (3, d)).astype(np.float32)
    res, _ = ctx.evaluate_swarm(gpu_params(S, "gini", 4, 3, 0, 16), wl.X, pos, labels=wl.labels,
                                sample_idx=idx, want_bins=True)
    ref, _, _ = O.eval_swarm(oracle_params(O, "gini", 4, 3, 0, 16), wl.X, wl.labels, None,
                             pos.astype(np.float64), idx=idx)
    for g, r in zip(res, ref):
        assert g["valid"] == r["valid"]
        for k in ("bin", "n_left", "n_right", "q_num", "q_den") if r["valid"] else ():
            assert g[k] == r[k], k
