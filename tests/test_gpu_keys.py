"""Small, mid and medium vertices keyed in one launch (csrc/kb_keys.cu), against
the oracle: sizes around a task and a block, with each class alone and all of
them with equal signatures across classes."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def check(g, **kw):
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    opts = kb.Options(**kw)
    L, C, _ = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=3, early_stop=False)
    for i in (1, 2, 3):
        prev = torch.from_numpy(L[i - 1].copy()).cuda()
        out = torch.empty_like(prev)
        assert kb.refine_round_noalloc(dg, prev, out, opts) == C[i]
        assert np.array_equal(out.cpu().numpy(), L[i]), (g.n, i, kw)


@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, 20_011])
@pytest.mark.parametrize("degrees", [[0, 1, 8], [9, 32], [33, 256], [257, 1024], [0, 2, 8, 9, 31, 32, 33, 200, 256, 257, 700, 1024]])
def test_classes_in_one_launch(n, degrees):
    rng = np.random.Generator(np.random.PCG64(n + len(degrees)))
    deg = rng.choice(degrees, size=n)
    if n > 1_000:  # large degrees are rare
        deg = np.where(rng.random(n) < 0.02, deg, np.minimum(deg, 9 if 9 in degrees else min(degrees)))
    src = np.repeat(np.arange(n), deg)
    # few targets for a third of the vertices: equal sets among all classes
    dst = rng.integers(0, 1 << 30, size=src.shape[0]) % np.minimum(n, rng.choice([1, 3, n], size=n))[src]
    g = graphgen.from_edges(n, src, dst, rng.integers(0, 2, size=src.shape[0]), rng.integers(0, 2, size=n))
    check(g)
    check(g, medium_split=100, small_max_degree=20, small_task_vertices=40)
