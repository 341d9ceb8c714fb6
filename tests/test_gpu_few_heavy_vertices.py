"""Small graphs of few vertices with many edges each: the kernel of all rounds
takes its CTAs by vertices or edges, whichever ask for more.  Against the oracle,
and not slower than the same call with one kernel per pass."""
import time

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def heavy(n, degree, targets, seed=0):
    rng = np.random.Generator(np.random.PCG64(seed))
    m = n * degree
    return graphgen.from_edges(n, np.repeat(np.arange(n), degree), rng.integers(0, targets, size=m),
                               rng.integers(0, 3, size=m), rng.integers(0, 3, size=n))


@pytest.mark.parametrize("n,degree", [(1, 1), (1, 1023), (1, 1025), (1, 200_000), (5, 1024), (256, 4), (257, 5),
                                      (300, 500), (1500, 1000), (700, 2900)])
def test_levels(n, degree):
    with kb.Context(0) as ctx:
        for targets in {1, min(n, 3), n}:
            g = heavy(n, degree, targets, seed=n + targets)
            dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
            for d in (kb.DIR_OUT, kb.DIR_IN):
                res = ctx.refine(dg, 4, kb.Options(direction=d))
                L, C, lc = oracle.refine_graph(g, d, True, True, k=4)
                assert np.array_equal(res.levels.cpu().numpy(), L[:5]) and np.array_equal(res.counts, C)
                assert res.levels_computed == lc


@pytest.mark.parametrize("n,degree", [(1500, 1000), (3000, 500)])
def test_not_slower_than_one_kernel_per_pass(n, degree):
    dg = kb.DeviceGraph.from_numpy(heavy(n, degree, n), "cuda:0")
    best = {}
    with kb.Context(0) as ctx:
        for ctas in (0, -1):
            ctx.set_round_kernel(max_ctas=ctas)
            ts = []
            for _ in range(20):
                torch.cuda.synchronize()
                t = time.perf_counter()
                ctx.refine(dg, 4)
                torch.cuda.synchronize()
                ts.append(time.perf_counter() - t)
            best[ctas] = min(ts)
    assert best[-1] < 1.5 * best[0], best
