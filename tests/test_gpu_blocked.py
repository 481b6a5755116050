"""The projection from blocked rows, not folded (the default where a batch is
long, has more nodes than CTAs, runs adaptive PSO or a swarm that does not
fold): the results of the row-major projection bit for bit. Swarm widths of
every particles-per-thread variant in long batches, short ones (narrow slices), slices cut
down because their positions would not fit, feature counts around the
16-feature chunks and odd ones, nodes smaller than a block, and levels of many
small nodes (several warps sharing a block)."""
import numpy as np
import pytest

from paper_2208_07023_gb300 import workloads as W
from tests.gpu_util import context, gpu_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctxs():
    a, b = context(), context()
    b.set_fused_step(False)
    yield a, b
    a.close()
    b.close()


@pytest.mark.parametrize("n,d,P,apso", [
    (3001, 17, 65, False),    # two slices of 40
    (2000, 16, 100, False),
    (700, 1, 256, False),     # four slices of 64, one feature
    (900, 1024, 70, False),   # slices cut to the positions' room
    (333, 300, 128, False),
    (31, 5, 80, False),       # less than one block
    (3000, 130, 250, False), (9000, 12, 100, False), (20011, 40, 250, False),
    # long: the fewest slices, of 5 to 8 particles a thread
    (90001, 3, 65, False), (90001, 4, 90, False), (90003, 17, 100, False), (90000, 5, 128, False),
    (90001, 3, 7, True), (90001, 5, 15, True), (70001, 3, 23, True), (70001, 3, 31, True),
    (70001, 3, 39, True), (70003, 3, 47, True), (70001, 6, 55, True), (70001, 3, 63, True),
    (5000, 23, 7, True), (4097, 33, 15, True), (2500, 50, 23, True), (2500, 48, 31, True),
    (1200, 15, 39, True), (1200, 31, 47, True), (800, 64, 55, True), (4100, 12, 63, True),
])
def test_search_identical_blocked_and_row_major(ctxs, n, d, P, apso):
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    wl = W.gmm(n, d, 3, seed=d + P)
    p = S.make_params("gini", 3, n_particles=P, n_iters=4, n_bins=64, min_leaf=2, seed=3,
                      apso=apso)
    before = a.set_fused_step(True)
    ra = a.node_split(p, wl.X, labels=wl.labels, node_uid=9, want_trace=True)
    assert a.set_fused_step(True) == before  # not folded
    rb = b.node_split(p, wl.X, labels=wl.labels, node_uid=9, want_trace=True)
    assert np.array_equal(ra["trace"], rb["trace"])
    assert np.array_equal(ra["gbest"].view(np.uint32), rb["gbest"].view(np.uint32))
    for k in ("bin", "q_num", "q_den", "n_left", "particle", "iter_of_best"):
        assert ra[k] == rb[k], k


@pytest.mark.parametrize("P,d", [(24, 9), (64, 20), (40, 33), (16, 6)])
def test_many_small_nodes_identical(ctxs, P, d):
    """More nodes than CTAs: runs of several nodes, 1, 2 or 4 warps a block."""
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    wl = W.tanh_regression(9000, d, seed=P)
    p = gpu_params(S, "mse", 0, P, 3, 64, min_leaf=4, max_depth=10, seed=2)
    ga, gb = (c.train_tree(p, wl.X, y=wl.y).export(0) for c in (a, b))
    for k in ga:
        assert np.array_equal(ga[k], gb[k]), k
    assert (ga["kind"] == 1).sum() > 500


@pytest.mark.parametrize("trees,n,P,d", [(2, 900, 72, 33), (5, 61, 100, 20), (17, 700, 250, 9),
                                         (40, 2000, 96, 130), (300, 200, 100, 7)])
def test_batches_of_short_nodes_identical(ctxs, trees, n, P, d):
    """Up to a few blocks a warp: narrow slices of several nodes."""
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    wl = W.gmm(n, d, 3, seed=P)
    p = gpu_params(S, "gini", 3, P, 3, 64, min_leaf=2, max_depth=2, seed=2, n_trees=trees,
                   bootstrap=True)
    fa, fb = (c.train_tree(p, wl.X, labels=wl.labels) for c in (a, b))
    for t in range(trees):
        ga, gb = fa.export(t), fb.export(t)
        for k in ga:
            assert np.array_equal(ga[k], gb[k]), (t, k)
    fa.free()
    fb.free()


@pytest.mark.parametrize("n,d,P,k", [
    (5000, 32, 64, 8),
    (3001, 17, 48, 8),    # odd feature count, a ragged last block
    (4099, 9, 40, 3),     # fewer than 8 re-scored
    (2500, 65, 64, 16),   # two slices
    (700, 8, 32, 20),     # three, the last of four
    (30, 5, 24, 8),       # less than one block
    (1500, 600, 32, 8),
])
@pytest.mark.parametrize("crit", ["gini", "mse"])
def test_bf16_rescores_identical(ctxs, crit, n, d, P, k):
    """The FP32 re-scores of the BF16 form from blocked rows (a thread takes
    two rows and eight particles): the row-major kernel's."""
    from paper_2208_07023_gb300 import binding as S
    a, b = ctxs
    if crit == "gini":
        wl = W.gmm(n, d, 4, seed=d)
        kw = dict(labels=wl.labels)
    else:
        wl = W.tanh_regression(n, d, seed=d)
        kw = dict(y=wl.y)
    p = S.make_params(crit, 4 if crit == "gini" else 0, n_particles=P, n_iters=4, n_bins=64,
                      min_leaf=2, seed=3, max_depth=4, proj=S.SLM_PROJ_BF16_TOPK, topk=k)
    ra, rb = (c.node_split(p, wl.X, node_uid=9, want_trace=True, **kw) for c in (a, b))
    assert np.array_equal(ra["trace"], rb["trace"])
    assert np.array_equal(ra["gbest"].view(np.uint32), rb["gbest"].view(np.uint32))
    assert ra["particle"] == rb["particle"] and ra["bin"] == rb["bin"]
    ga, gb = (c.train_tree(p, wl.X, **kw).export(0) for c in (a, b))
    for key in ga:
        assert np.array_equal(ga[key], gb[key]), key
