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


@pytest.mark.parametrize("polls", [1, 40])
@pytest.mark.parametrize("labels", [True, False])
def test_calls_start_again_when_a_wait_runs_out(polls, labels):
    g = graph(100_000, 300_000, 3)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    opts = kb.Options(use_vertex_labels=labels)
    L, C, lc = oracle.refine_graph(g, kb.DIR_OUT, labels, True, k=70)
    full, _, _ = oracle.refine_graph(g, kb.DIR_OUT, labels, True, k=70, early_stop=False)
    with kb.Context(0) as ctx:
        ctx.set_round_kernel(max_polls=polls)
        check(ctx.refine(dg, 5, opts), g, 5, opts)
        assert ctx.round_kernel() == (1, 0, 1)
        check(ctx.refine(dg, 70, kb.Options(use_vertex_labels=labels, early_stop=False)), g, 70,
              kb.Options(use_vertex_labels=labels, early_stop=False))
        final, count, rounds, stable = ctx.refine_fixpoint(dg, 70, opts)
        assert np.array_equal(final.cpu().numpy(), full[70]) and (count, rounds, stable) == (C[70], lc, True)
        host = ctx.refine_host(g.row_offsets, g.col, g.elabel, g.vlabel, 5, opts)
        assert np.array_equal(host.levels, L[:6]) and np.array_equal(host.counts, C[:6])
        with ctx.prepare(dg, kb.Options(use_vertex_labels=labels, reorder=2)) as pg:
            check(ctx.refine(pg, 5), g, 5, opts)
        # starts that are a row of the levels: the starting one, a later one, another array
        for src in (1, 3, None):
            rows = torch.zeros((6, g.n), dtype=torch.int32, device="cuda:0")
            start = rows[src] if src is not None else torch.empty_like(rows[0])
            start.copy_(torch.from_numpy(7 * L[1]))
            res = ctx.refine_from(dg, start, 1, 5, opts, levels=rows)
            assert np.array_equal(res.levels[1:].cpu().numpy(), L[1:6]) and np.array_equal(res.counts[1:], C[1:6])
        launches, refused, gave_up = ctx.round_kernel()
        assert refused == 0 and launches == gave_up == 8


def test_calls_start_again_when_the_launch_is_refused():
    g = graph(900_000, 900_000, 1)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    with kb.Context(0) as ctx:
        ctx.set_round_kernel(max_ctas=1 << 20)  # more CTAs than a device holds at once
        check(ctx.refine(dg, 4), g, 4)
        assert ctx.round_kernel() == (0, 1, 0)
        ctx.set_round_kernel()
        check(ctx.refine(dg, 4), g, 4)
        assert ctx.round_kernel() == (1, 1, 0)


def test_a_phase_longer_than_the_wait():
    # one previous block, all signatures distinct, hashes equal: every insertion walks the chain of those before it
    n = 520_000
    rng = np.random.Generator(np.random.PCG64(5))
    g = graphgen.from_edges(n, np.repeat(np.arange(n), 3), rng.integers(0, n, size=3 * n),
                            rng.integers(0, 1 << 30, size=3 * n))
    opts = kb.Options.schaetzle(hash_mode=1)
    with kb.Context(0) as ctx:
        check(ctx.refine(kb.DeviceGraph.from_numpy(g, "cuda:0"), 1, opts), g, 1, opts)
