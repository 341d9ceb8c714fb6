"""Tiles of edges whose sources lie far apart: runs of edgeless vertices (or of
empty graphs in a batch) around the length from which a tile searches for its
sources instead of walking them, through the in-edge CSR, the summary graph and
the batch's graph ids.  Against the oracle, and not slower than the same edges
side by side."""
import time

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

WALK = 8  # vertices per edge of a tile
TILES = (1024, 2048)  # summary; in-edge CSR and graph ids


@pytest.fixture(scope="module")
def ctx():
    c = kb.Context(0)
    yield c
    c.close()


def gapped(n, m, gap, seed):
    """m edges among n vertices, of which the upper half lies `gap` edgeless vertices behind the lower one."""
    rng = np.random.Generator(np.random.PCG64(seed))
    src, dst = rng.integers(0, n, size=m), rng.integers(0, n + gap, size=m)
    return graphgen.from_edges(n + gap, np.where(src >= n // 2, src + gap, src), dst, rng.integers(0, 3, size=m),
                               rng.integers(0, 4, size=n + gap))


@pytest.mark.parametrize("gap", sorted({WALK * t + x for t in TILES for x in (-3, -2, -1, 0, 1)} | {0, 300_000}))
def test_gaps(ctx, gap):
    for n, m in ((2, 900), (2, 2048), (3, 2049), (40, 5000), (3000, 7001)):
        g = gapped(n, m, gap, seed=n + gap)
        dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
        for d in (kb.DIR_IN, kb.DIR_BOTH):
            res = ctx.refine(dg, 2, kb.Options(direction=d))
            L, C, _ = oracle.refine_graph(g, d, True, True, k=2)
            assert np.array_equal(res.levels.cpu().numpy(), L[:3]) and np.array_equal(res.counts, C), (n, d)
        a, b = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (L[2], L[1]))
        for d in (kb.DIR_OUT, kb.DIR_IN):
            for got, want in zip(ctx.summary(dg, a, b, direction=d), oracle.summary(g, d, True, L[2], L[1])):
                assert np.array_equal(got.cpu().numpy(), want), (n, d)


@pytest.mark.parametrize("empty", [0, WALK * 2048 - 1, WALK * 2048, WALK * 2048 + 1, 100_000])
def test_empty_graphs_of_a_batch(ctx, empty):
    gs = [graphgen.erdos_renyi(n, 3 * n, 3, 2, seed=n) for n in (700, 1, 900, 2500)]
    sizes = np.concatenate([[gs[0].n], np.zeros(empty, dtype=np.int64), [g.n for g in gs[1:]]])
    voff = np.concatenate([[0], np.cumsum(sizes)])
    union, _ = graphgen.disjoint_union(gs)
    levels, counts, _ = ctx.refine_batch(kb.DeviceGraph.from_numpy(union, "cuda:0"), voff,
                                         np.full(len(sizes), 3, dtype=np.int32))
    levels = levels.cpu().numpy()
    for j, g in zip([0] + list(range(empty + 1, empty + len(gs))), gs):
        L, C, _ = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=3)
        assert np.array_equal(levels[:, voff[j]:voff[j + 1]], L[:4]) and np.array_equal(counts[j], C), j
    assert not counts[1:empty + 1].any()


def test_long_runs_cost_little(ctx):
    def best(gap):
        g = gapped(2_000_000, 1_000_000, gap, seed=1)
        dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
        lv = ctx.refine(dg, 1, kb.Options()).levels
        ts = []
        for _ in range(12):
            torch.cuda.synchronize()
            t = time.perf_counter()
            ctx.summary(dg, lv[1], lv[0])
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t)
        return min(ts)

    # the tile that walked the run took thousands of microseconds; the run itself adds some 20 to the offsets' check
    assert best(4_000_000) < 4 * best(0)
