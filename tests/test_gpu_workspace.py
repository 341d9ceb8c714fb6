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
