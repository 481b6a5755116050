"""Regression scores from the 30-bit rounded targets (mse_kernels.cu) are those
of the staged-copy kernel, bit for bit: an edge's rounded interval may only
rule it out, and every edge left is scored exactly. Sizes at the edges of the
kernels: the largest warp node (2,048 entries) and the smallest cluster node,
slices around the switch from 8 to 32 copies per bin, the largest slice of a
single CTA, bins per lane of every width, targets that leave many edges
(two values, one value, one far outlier), and targets that are not finite."""
import numpy as np
import pytest

from paper_2208_07023_gb300 import workloads as W
from tests.gpu_util import context, gpu_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctxs():
    a, b = context(), context()
    b.set_class_hist(False)  # the staged-copy kernel scores every particle
    yield a, b
    a.set_small_nodes()
    a.close()
    b.close()


def _targets(kind, wl):
    y = wl.y.copy()
    if kind == "two":
        return (y > 0.3).astype(np.float32) * 0.9 - 0.1
    if kind == "one":
        return np.full_like(y, 0.25)
    if kind == "outlier":
        y[len(y) // 2] = 3e6
    if kind == "offset":
        y = (y * np.float32(1e-3) + np.float32(500)).astype(np.float32)
    if kind == "crowd":  # nearly all at the largest rounded target, 2^28 - 1
        y = np.full_like(y, 0.4999999)
        y[::1000] = -0.4999999
    if kind in ("inf", "-inf", "nan", "infs"):
        y[len(y) // 3] = {"-inf": -np.inf, "nan": np.nan}.get(kind, np.inf)
    if kind == "infs":
        y[:len(y) // 2:3] = -np.inf
    return y


def _same_search(a, b, p, X, y):
    ra = a.node_split(p, X, y=y, node_uid=8, want_trace=True)
    rb = b.node_split(p, X, y=y, node_uid=8, want_trace=True)
    assert np.array_equal(ra["trace"], rb["trace"], equal_nan=True)
    assert np.array_equal(ra["gbest"].view(np.uint32), rb["gbest"].view(np.uint32))
    for k in ("valid", "bin", "loss", "n_left", "n_right", "particle", "iter_of_best"):
        assert ra[k] == rb[k] or (k == "loss" and np.isnan(ra[k]) and np.isnan(rb[k])), k


@pytest.mark.parametrize("n,B,min_leaf,kind", [
    (2048, 256, 1, "plain"), (2049, 256, 1, "plain"), (2047, 200, 5, "plain"),
    (65, 33, 1, "plain"), (3, 16, 1, "plain"), (700, 2, 1, "plain"),
    (1500, 64, 1, "two"), (1500, 100, 1, "one"), (1800, 256, 1, "outlier"),
    (1900, 128, 3, "offset"), (8190, 32, 1, "two"), (9000, 256, 1, "one"),
    (40001, 256, 5, "plain"), (40001, 256, 1, "outlier"), (70003, 128, 1, "offset"),
    (131003, 256, 20, "plain"),
])
@pytest.mark.parametrize("warp", [False, True])
def test_search_identical_to_the_exact_histogram(ctxs, n, B, min_leaf, kind, warp):
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    a.set_small_nodes(4096 if warp else 0, 0)
    wl = W.tanh_regression(n, 6, seed=n % 83)
    y = _targets(kind, wl)
    p = gpu_params(S, "mse", 0, 19, 9, B, min_leaf=min_leaf, seed=3)
    _same_search(a, b, p, wl.X, y)


@pytest.mark.parametrize("n,B,kind", [(700, 32, "inf"), (701, 64, "nan"), (1999, 256, "infs"),
                                      (9000, 128, "-inf"), (9001, 256, "inf"),
                                      (20000, 200, "infs"), (20000, 200, "nan")])
@pytest.mark.parametrize("warp", [False, True])
def test_targets_that_are_not_finite(ctxs, n, B, kind, warp):
    """No bound follows from them: every edge is scored."""
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    a.set_small_nodes(4096 if warp else 0, 0)
    wl = W.tanh_regression(n, 6, seed=n % 83)
    p = gpu_params(S, "mse", 0, 19, 9, B, min_leaf=2, seed=3)
    _same_search(a, b, p, wl.X, _targets(kind, wl))


# 250 particles: a CTA per particle as long as the node fits its counters
@pytest.mark.parametrize("n,B,kind,S_want", [
    (8188, 256, "plain", 1),   # the longest slice of 8 copies
    (8189, 256, "plain", 1),   # 32 copies from here on
    (20001, 200, "two", 1),
    (30011, 100, "offset", 1),
    (64996, 256, "plain", 1),  # the largest slice: 2,032 of 2,048 entries a copy
    (64995, 32, "crowd", 1),   # and sums of the high words near 2^32 in one bin
    (64996, 2, "crowd", 1),
    (64997, 64, "outlier", 2),
])
def test_long_slices_identical_to_the_exact_histogram(ctxs, n, B, kind, S_want):
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    a.set_small_nodes(0, 0)
    wl = W.tanh_regression(n, 6, seed=n % 83)
    X = wl.X
    if kind == "crowd":  # one far row: the others share a bin
        X = X.copy()
        X[0] *= 1e4
    p = gpu_params(S, "mse", 0, 250, 4, B, min_leaf=1, seed=3)
    _same_search(a, b, p, X, _targets(kind, wl))
    a.node_split(p, X, y=_targets(kind, wl), node_uid=8)
    assert a.tuning_stats()["last_hist_cluster"] == S_want


@pytest.mark.parametrize("d,P", [(6, 64), (400, 64), (400, 19)])
def test_slices_are_one_wave(ctxs, d, P):
    """Rows of 400 features leave room for two CTAs per SM, not three."""
    import torch
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    a.set_small_nodes()
    n = 131000
    g = torch.Generator(device="cuda").manual_seed(d)
    X = torch.randn(n, d, generator=g, device="cuda")
    y = torch.tanh(X[:, 0] + X[:, 1]) + 0.1 * torch.randn(n, generator=g, device="cuda")
    p = gpu_params(S, "mse", 0, P, 2, 256, min_leaf=5, seed=3)
    _same_search(a, b, p, X, y)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    assert a.tuning_stats()["last_hist_cluster"] * P <= (2 if d == 400 else 3) * n_sm


@pytest.mark.parametrize("proj,apso", [("fp32", False), ("bf16", False), ("fp32", True)])
def test_tree_identical_to_the_exact_histogram(ctxs, proj, apso):
    """Levels of hundreds of small nodes (a warp each), beside large ones."""
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    a.set_small_nodes()
    wl = W.tanh_regression(12000, 9, seed=5)
    p = S.make_params("mse", 0, n_particles=24, n_iters=6, n_bins=200, min_leaf=4, max_depth=9,
                      seed=5, proj=S.SLM_PROJ_BF16_TOPK if proj == "bf16" else S.SLM_PROJ_FP32,
                      topk=5, apso=apso)
    ga, gb = (c.train_tree(p, wl.X, y=wl.y).export(0) for c in (a, b))
    for k in ga:
        assert np.array_equal(ga[k], gb[k]), k
    assert (ga["kind"] == 1).sum() > 200
