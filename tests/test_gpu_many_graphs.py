"""Batches around the number of graphs from which their offsets and k go to the
device from where they lie instead of through one staged copy.  Against the oracle
on the template that the batch repeats."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

STAGE = 512 << 10  # bytes of offsets (8), k (4), active (1) and last level (4)


@pytest.mark.parametrize("G", [1, 2, 7, STAGE // 17 - 60, STAGE // 17 + 60, 200_000])
def test_levels(G):
    parts = [graphgen.path_graph(4), graphgen.cycle_graph(3), graphgen.erdos_renyi(5, 9, 2, 2, seed=1)]
    template, _ = graphgen.disjoint_union(parts)
    reps = -(-G // 3)
    sizes = np.tile([p.n for p in parts], reps)[:G]
    voff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(voff[-1])
    deg = np.tile(np.diff(template.row_offsets), reps)[:n]
    row = np.concatenate([[0], np.cumsum(deg)])
    m = int(row[-1])
    first = np.repeat(voff[:-1], sizes)  # first vertex of every vertex's graph
    local = np.concatenate([p.col for p in parts])
    union = graphgen.Graph(n=n, m=m, row_offsets=row, col=(np.tile(local, reps)[:m] + np.repeat(first, deg)).astype(np.int32),
                           elabel=np.tile(template.elabel, reps)[:m], vlabel=np.tile(template.vlabel, reps)[:n], names=None)
    ks = (np.arange(G) % 4).astype(np.int32)
    with kb.Context(0) as ctx:
        levels, counts, computed = ctx.refine_batch(kb.DeviceGraph.from_numpy(union, "cuda:0"), voff, ks)
    levels = levels.cpu().numpy()
    kmax = int(ks.max())
    for j in range(min(3, G)):
        g = parts[j]
        for k in range(4):
            mine = [i for i in range(j, G, 3) if ks[i] == k]
            if not mine:
                continue
            L, C, lc = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=k)
            at = np.asarray(mine)
            for i in range(kmax + 1):
                want = L[min(i, k)]
                got = levels[i][voff[at][:, None] + np.arange(g.n)]
                assert (got == want).all(), (j, k, i)
                assert (counts[at, i] == C[min(i, k)]).all()
            assert (computed[at] == lc).all()
