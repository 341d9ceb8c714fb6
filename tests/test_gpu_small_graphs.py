"""Work splits and launch rules of small graphs, against the oracle.

Warp tasks, medium tasks and the tiles that refill the hub sets get shorter
while a graph is too small to fill the chip: vertex counts around the edges of
a task and of a window, with the rounds on packed windows (most vertices
frozen) and on long sparse tasks among them.
"""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


@pytest.fixture(scope="module")
def ctx():
    c = kb.Context(0)
    yield c
    c.close()


def check(ctx, g, d, k, prepared=False, **kw):
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    opts = kb.Options(direction=d, **kw)
    if prepared:
        with ctx.prepare(dg, opts) as pg:
            res = ctx.refine(pg, k)
    else:
        res = ctx.refine(dg, k, opts)
    L, C, lc = oracle.refine_graph(g, d, opts.use_vertex_labels, opts.use_edge_labels, k=k, early_stop=opts.early_stop)
    got = res.levels.cpu().numpy()
    for i in range(k + 1):
        assert np.array_equal(got[i], L[i]), (g.n, d, kw, "level %d" % i)
    assert np.array_equal(res.counts, C) and res.levels_computed == lc


@pytest.mark.parametrize("n", [1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 255, 256, 257, 116_735, 116_737])
def test_sizes_around_tasks_and_windows(ctx, n):
    for m, labels in ((0, 2), (3 * n, 3), (5 * n + 1, n // 4 + 1)):
        g = graphgen.erdos_renyi(n, m, labels, 2, seed=n)
        for d in (kb.DIR_OUT, kb.DIR_BOTH):
            check(ctx, g, d, 5, early_stop=False)
            check(ctx, g, d, 5, prepared=True, reorder=2)


@pytest.mark.parametrize("n", [300, 5_000, 200_003])
def test_sparse_rounds(ctx, n):
    # a long path behind labelled singletons: after the first rounds only the
    # path's vertices refine, a few per round
    tail = 200
    src = np.concatenate([np.arange(n), n + np.arange(tail)])
    dst = np.concatenate([np.arange(n), np.minimum(n + np.arange(tail) + 1, n + tail - 1)])
    vl = np.concatenate([np.arange(n) + 1, np.zeros(tail, dtype=np.int64)])
    vl[n + tail - 1] = n + 5
    g = graphgen.from_edges(n + tail, src, dst, None, vl)
    check(ctx, g, kb.DIR_OUT, 40)


@pytest.mark.parametrize("n_medium,n_hubs", [(1, 0), (5, 1), (700, 3), (9_000, 0)])
def test_few_medium_vertices_and_hubs(ctx, n_medium, n_hubs):
    rng = np.random.Generator(np.random.PCG64(n_medium))
    n = 10_000
    deg = rng.integers(0, 4, size=n)
    deg[:n_medium] = rng.choice([33, 34, 200, 256, 257, 300, 1024], size=n_medium)
    deg[n - n_hubs:] = 1025 + rng.integers(0, 3000, size=n_hubs)
    src = np.repeat(np.arange(n), deg)
    # targets repeat with the degree, so that equal signatures occur among medium vertices
    dst = (np.arange(src.shape[0]) * 7) % 23 if n_medium < 700 else rng.integers(0, 40, size=src.shape[0])
    g = graphgen.from_edges(n, src, dst, rng.integers(0, 2, size=src.shape[0]), rng.integers(0, 2, size=n))
    check(ctx, g, kb.DIR_OUT, 4, early_stop=False)
    check(ctx, g, kb.DIR_IN, 4, early_stop=False)
