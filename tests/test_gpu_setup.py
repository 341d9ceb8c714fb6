"""Setup of a call (csrc/kb_setup.cu), against the oracle: hubs handed out as they
are found or listed, tile counts in the counters or in the scratch, ids checked
beside the degree classes, and label minima left empty for the next call."""
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


def check(ctx, g, k=3, **kw):
    opts = kb.Options(**kw)
    res = ctx.refine(kb.DeviceGraph.from_numpy(g, "cuda:0"), k, opts)
    L, C, _ = oracle.refine_graph(g, opts.direction, True, True, k=k)
    assert np.array_equal(res.levels.cpu().numpy(), L) and np.array_equal(res.counts, C)


# at most 4096 hubs fit the buffer that takes them as they are found
@pytest.mark.parametrize("thr,m", [(8, 9 * 4095), (8, 9 * 4096 - 1), (8, 9 * 4096), (8, 9 * 4400), (40, 60_000)])
def test_hubs_found_or_listed(ctx, thr, m):
    deg = np.full(5_000, 0)
    deg[: m // 12] = 12  # as many hubs as the edges give, of 9 and more edges
    deg[7] += m - deg.sum()
    src = np.repeat(np.random.Generator(np.random.PCG64(m)).permutation(5_000), deg)
    rng = np.random.Generator(np.random.PCG64(m + 1))
    g = graphgen.from_edges(5_000, src, rng.integers(0, 40, size=m), rng.integers(0, 2, size=m), rng.integers(0, 3, size=5_000))
    check(ctx, g, hub_threshold=thr)


@pytest.mark.parametrize("n", [131_071, 131_072, 32 * 131_072, 32 * 131_072 + 1])
def test_tiles_of_the_class_lists(ctx, n):
    rng = np.random.Generator(np.random.PCG64(n))
    big = rng.choice(n, size=300, replace=False)  # mid and medium vertices in the first and last tiles too
    big[:4] = (0, n - 1, n // 2, n - 2)
    src = np.repeat(big, rng.choice([9, 32, 33, 200], size=300))
    g = graphgen.from_edges(n, src, rng.integers(0, n, size=src.shape[0]), None, rng.integers(0, 5, size=n))
    check(ctx, g, k=2)


@pytest.mark.parametrize("m", [1, 255, 256, 257, 5_000, 8 * 256 * 152 * 16 + 3])
def test_ids_out_of_range(ctx, m):
    n = 1_000
    g = graphgen.erdos_renyi(n, m, 2, 2, seed=m)
    check(ctx, g, k=1)
    for at, wrong in ((0, -1), (m - 1, n), (m // 2, 2**31 - 1)):
        col = g.col.copy()
        col[at] = wrong
        dg = kb.DeviceGraph(*(torch.from_numpy(x).cuda() for x in (g.row_offsets, col, g.elabel, g.vlabel)))
        with pytest.raises(kb.KbError):
            ctx.refine(dg, 1, kb.Options())
    check(ctx, g, k=1)


def test_small_and_large_labels_in_turn(ctx):
    rng = np.random.Generator(np.random.PCG64(1))
    for n_labels in (3, 9_000, 8_192, 20_000, 5, 8_193, 2):
        g = graphgen.erdos_renyi(20_000, 30_000, 2, 2, seed=n_labels)
        g.vlabel[:] = rng.integers(0, n_labels, size=20_000)
        g.vlabel[0] = n_labels - 1
        check(ctx, g, early_stop=True)
