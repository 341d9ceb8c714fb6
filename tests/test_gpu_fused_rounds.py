"""All rounds of a small graph in one kernel (csrc/kb_fused.cu), against the
oracle and against the same call with a launch per pass (which per-round timing
selects): sizes around the rule's limit and around the rank scan's two forms,
more rounds than one launch runs, hubs of every chunk size beside medium
vertices, and a start from a given level."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

LIMIT = 1 << 21  # vertices and processed edges


@pytest.fixture(scope="module")
def ctx():
    c = kb.Context(0)
    yield c
    c.close()


def check(ctx, g, k, **kw):
    opts = kb.Options(**kw)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    L, C, lc = oracle.refine_graph(g, opts.direction, opts.use_vertex_labels, opts.use_edge_labels, k=k,
                                   early_stop=opts.early_stop)
    for timing in (False, True, False):
        ctx.set_timing(timing)
        res = ctx.refine(dg, k, opts)
        assert np.array_equal(res.levels.cpu().numpy(), L[:k + 1]), timing
        assert np.array_equal(res.counts, C) and res.levels_computed == lc, timing
    ctx.set_timing(False)
    host = ctx.refine_host(g.row_offsets, g.col, g.elabel, g.vlabel, k, opts)
    assert np.array_equal(host.levels, L[:k + 1]) and np.array_equal(host.counts, C)
    return L, C


@pytest.mark.parametrize("n,extra,d", [
    (400_000, -1, kb.DIR_OUT), (400_000, 0, kb.DIR_OUT), (400_000, 1, kb.DIR_OUT),
    (500_000, 0, kb.DIR_BOTH), (16_384 * 32 - 32, 0, kb.DIR_IN), (16_384 * 32 - 1, 0, kb.DIR_IN),
    (16_384 * 32, 0, kb.DIR_IN), (2_000_000, 0, kb.DIR_IN)])
def test_sizes_around_the_limits(ctx, n, extra, d):
    m = (LIMIT - n + extra) // (2 if d == kb.DIR_BOTH else 1)
    check(ctx, graphgen.erdos_renyi(n, m, 5, 2, seed=n + extra), 4, direction=d)


@pytest.mark.parametrize("length,k", [(63, 64), (64, 65), (64, 64), (130, 200), (300, 150)])
def test_more_rounds_than_a_launch_runs(ctx, length, k):
    g = graphgen.path_graph(length)
    for stop in (True, False):
        check(ctx, g, k, early_stop=stop, use_vertex_labels=False)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    opts = kb.Options(use_vertex_labels=False)
    want = oracle.refine_graph(g, opts.direction, False, True, k=k)
    final, count, rounds, _ = ctx.refine_fixpoint(dg, k, opts)
    assert np.array_equal(final.cpu().numpy(), want[0][k]) and count == want[1][k] and rounds == want[2]
    # an epoch of the block table per round: many calls pass its limit in mid-launch
    for _ in range(6):
        assert torch.equal(ctx.refine_fixpoint(dg, k, opts)[0], final)


@pytest.mark.parametrize("chunk,thr,split", [(256, 300, 100), (512, 0, 0), (1024, 1024, 256), (1024, 64, 0)])
@pytest.mark.parametrize("d", [kb.DIR_OUT, kb.DIR_BOTH])
def test_hubs_and_medium_vertices(ctx, chunk, thr, split, d):
    rng = np.random.Generator(np.random.PCG64(chunk + thr))
    n = 6_000
    deg = rng.choice([0, 1, 3, 8, 9, 20, 32, 33, 100, 256, 257, 700, 1024, 1025, 5000], size=n,
                     p=[.2, .2, .2, .1, .1, .05, .05, .03, .02, .01, .01, .01, .01, .007, .003])
    src = np.repeat(np.arange(n), deg)
    # a vertex's edges reach few or many targets, so that equal signatures occur in every class
    dst = rng.integers(0, 1 << 30, size=src.shape[0]) % rng.choice([2, 9, n], size=n)[src]
    g = graphgen.from_edges(n, src, dst, rng.integers(0, 2, size=src.shape[0]), rng.integers(0, 3, size=n))
    for stop in (True, False):
        check(ctx, g, 6, direction=d, hub_chunk_edges=chunk, hub_threshold=thr, medium_split=split, early_stop=stop)


def test_from_a_given_level(ctx):
    g = graphgen.erdos_renyi(20_000, 70_000, 2, 2, seed=3)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    L, C, _ = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=6, early_stop=False)
    for opts in (kb.Options(early_stop=False), kb.Options(early_stop=False, reorder=2)):
        for i in (0, 2, 5):
            res = ctx.refine_from(dg, torch.from_numpy(L[i].copy()).cuda(), i, 6, opts)
            assert np.array_equal(res.levels[i:].cpu().numpy(), L[i:7])
            assert np.array_equal(res.counts[i:], C[i:7])
