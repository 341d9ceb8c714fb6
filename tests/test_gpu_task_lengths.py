"""Rounds in which few vertices refine, with a task length given by the caller:
the packed windows of the small graphs' kernel address a vertex within its task
in 16 bits, so a task may not grow past 65,536 vertices.  Against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def late_tail(n, tail):
    """n vertices alone in their blocks from the start and a path behind them, with consecutive ids past the
    others': only the path's vertices refine, more of them side by side than a window holds."""
    src = np.concatenate([np.arange(n), n + np.arange(tail)])
    dst = np.concatenate([np.arange(n), np.minimum(n + np.arange(tail) + 1, n + tail - 1)])
    vl = np.concatenate([np.arange(n) + 1, np.zeros(tail, dtype=np.int64)])
    vl[n + tail - 1] = n + 5
    return graphgen.from_edges(n + tail, src, dst, None, vl)


@pytest.mark.parametrize("n,tail", [(65_500, 200), (70_000, 20), (200_003, 200), (262_100, 900), (900_000, 200)])
def test_long_tasks(n, tail):
    g = late_tail(n, tail)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    L, C, lc = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=6)
    with kb.Context(0) as ctx:
        for task in (1_024, 4_095, 16_384, 16_385, 32_768, 65_536):
            res = ctx.refine(dg, 6, kb.Options(small_task_vertices=task))
            assert np.array_equal(res.levels.cpu().numpy(), L[:7]), task
            assert np.array_equal(res.counts, C) and res.levels_computed == lc, task
