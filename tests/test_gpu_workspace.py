"""Caller-owned scratch (kb_set_workspace): at any address that is a multiple of
eight bytes, and of the queried size for every graph of the queried size.  Against
the oracle."""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def hub_graph(n, m, hub_degree, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    src = np.concatenate([rng.integers(0, n, size=m), np.full(hub_degree, n // 2), np.full(hub_degree, n // 3)])
    return graphgen.from_edges(n, src, rng.integers(0, n, size=src.shape[0]), rng.integers(0, 3, size=src.shape[0]),
                               rng.integers(0, 3, size=n))


@pytest.mark.parametrize("offset", [0, 8, 24, 256])
@pytest.mark.parametrize("n,m,hub", [(33, 90, 0), (5_000, 20_000, 0), (5_000, 20_000, 3_000), (400_000, 2_000_000, 30_000)])
def test_any_eight_byte_address(offset, n, m, hub):
    g = hub_graph(n, m, hub, seed=n)
    dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
    with kb.Context(0) as ctx:
        for d in (kb.DIR_OUT, kb.DIR_BOTH):
            opts = kb.Options(direction=d)
            need = ctx.workspace_size(dg, 4, opts)
            buf = torch.empty(need + 1024, dtype=torch.uint8, device="cuda:0")
            at = buf.data_ptr() + (-buf.data_ptr()) % 256 + offset
            ctx._check(ctx._lib.kb_set_workspace(ctx._h, ctypes.c_void_p(at), need))
            L, C, lc = oracle.refine_graph(g, d, True, True, k=4)
            for early in (True, False):
                opts = kb.Options(direction=d, early_stop=early)
                L, C, lc = oracle.refine_graph(g, d, True, True, k=4, early_stop=early)
                res = ctx.refine(dg, 4, opts)
                assert np.array_equal(res.levels.cpu().numpy(), L[:5]) and np.array_equal(res.counts, C)
                assert res.levels_computed == lc
            torch.cuda.synchronize()
            ctx._check(ctx._lib.kb_set_workspace(ctx._h, None, 0))


@pytest.mark.parametrize("d", [kb.DIR_OUT, kb.DIR_IN, kb.DIR_BOTH])
def test_graph_changed_in_place(d):
    # the same tensors, vertices and edges; no vertex above eight edges, then some of 30 and of 200
    n, m = 20_000, 60_000
    few = graphgen.from_edges(n, np.arange(m) % n, (np.arange(m) * 7 + 1) % n, np.arange(m) % 3, np.arange(n) % 4)
    deg = np.zeros(n, dtype=np.int64)
    deg[:1_600] = 30
    deg[1_600:1_660] = 200
    src = np.repeat(np.arange(n), deg)
    rng = np.random.Generator(np.random.PCG64(2))
    ends = np.repeat(np.arange(n), deg[::-1])  # in-degrees of the same kind
    many = graphgen.from_edges(n, src, rng.permutation(ends), rng.integers(0, 3, size=m), np.arange(n) % 4)
    dg = kb.DeviceGraph.from_numpy(few, "cuda:0")
    opts = kb.Options(direction=d)
    with kb.Context(0, torch_workspace=True) as ctx:
        for g in (few, many, few):
            for t, a in ((dg.row_offsets, g.row_offsets), (dg.col, g.col), (dg.elabel, g.elabel), (dg.vlabel, g.vlabel)):
                t.copy_(torch.from_numpy(a))
            res = ctx.refine(dg, 4, opts)
            L, C, _ = oracle.refine_graph(g, d, True, True, k=4)
            assert np.array_equal(res.levels.cpu().numpy(), L[:5]) and np.array_equal(res.counts, C)
