"""The kernel of small graphs whose CTAs wait for one another, with its limits
set (kb_set_round_kernel): waits that run out, and the context's calls after."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

TIMEOUT = 4  # KB_ERR_TIMEOUT


def graph(n, m, shift, seed=11):
    """Labels 0..9 in ten runs of vertices, starting with label `shift`: every label's smallest vertex moves with it."""
    g = graphgen.erdos_renyi(n, m, 1, 3, seed=seed)
    return graphgen.from_edges(n, np.repeat(np.arange(n), np.diff(g.row_offsets)), g.col, g.elabel,
                               (np.arange(n) * 10 // n + shift) % 10)


def check(res, g, k, opts=None):
    opts = opts or kb.Options()
    L, C, lc = oracle.refine_graph(g, opts.direction, opts.use_vertex_labels, opts.use_edge_labels, k=k,
                                   early_stop=opts.early_stop)
    assert np.array_equal(res.levels.cpu().numpy(), L[:k + 1])
    assert np.array_equal(res.counts, C) and res.levels_computed == lc


@pytest.mark.parametrize("polls", [1, 3, 300])
def test_context_is_usable_after_a_wait_that_ran_out(polls):
    with kb.Context(0) as ctx:
        for rep in range(3):
            for prepared in (False, True):
                first, then = graph(100_000, 300_000, rep), graph(100_000, 300_000, rep + 4, seed=rep)
                dg, dt = kb.DeviceGraph.from_numpy(first, "cuda:0"), kb.DeviceGraph.from_numpy(then, "cuda:0")
                ctx.set_round_kernel(max_polls=polls)
                try:
                    if prepared:
                        with ctx.prepare(dg, kb.Options(reorder=2)) as pg:
                            check(ctx.refine(pg, 5), first, 5)
                    else:
                        check(ctx.refine(dg, 5), first, 5)
                except kb.KbError as e:
                    assert e.status == TIMEOUT
                ctx.set_round_kernel()
                check(ctx.refine(dt, 5), then, 5)
                check(ctx.refine(dg, 5), first, 5)


def test_without_it():
    g = graph(50_000, 200_000, 2)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    with kb.Context(0) as ctx:
        ctx.set_round_kernel(max_ctas=0, max_polls=1)
        check(ctx.refine(dg, 5), g, 5)
        ctx.set_round_kernel(max_ctas=7)
        check(ctx.refine(dg, 5), g, 5)
        with pytest.raises(kb.KbError):
            ctx.set_round_kernel(max_ctas=-2)
        with pytest.raises(kb.KbError):
            ctx.set_round_kernel(max_polls=-1)
