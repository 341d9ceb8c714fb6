"""Requests whose pinned arrays lie at any address, as slices of one buffer do:
those that a kernel's loads could not take are copied, as all were before pinned
arrays were read in place.  Against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def pinned_at(a, offset):
    """A pinned copy of a, `offset` bytes past an aligned address."""
    buf = torch.zeros(a.nbytes + 64, dtype=torch.uint8, pin_memory=True).numpy()
    out = np.frombuffer(buf.data, dtype=a.dtype, count=a.size, offset=(-buf.ctypes.data % 16) + offset)
    out[:] = a
    assert out.ctypes.data % 16 == offset
    return out


@pytest.mark.parametrize("offsets", [(0, 0, 0, 0), (8, 4, 12, 4), (4, 0, 0, 0), (0, 2, 0, 0), (0, 0, 1, 0), (0, 0, 0, 3),
                                     (7, 5, 3, 1)])
@pytest.mark.parametrize("d", [kb.DIR_OUT, kb.DIR_IN])
def test_any_address(offsets, d):
    with kb.Server(0, max_vertices=1 << 18, max_edges=1 << 20, max_requests=4) as server:
        jobs = []
        for n in (1, 700, 20_001):
            g = graphgen.erdos_renyi(n, 3 * n, 4, 3, seed=n)
            host = [pinned_at(a, o) for a, o in zip((g.row_offsets, g.col, g.elabel, g.vlabel), offsets)]
            out = pinned_at(np.zeros(5 * n, dtype=np.int32), offsets[1]).reshape(5, n)
            jobs.append((server.submit(*host, 4, kb.Options(direction=d), out=out), g, host))
        while any(server.step()):
            pass
        for ticket, g, _ in jobs:
            levels, counts, computed = server.fetch(ticket)
            L, C, lc = oracle.refine_graph(g, d, True, True, k=4)
            assert np.array_equal(levels, L[:5]) and np.array_equal(counts, C) and computed == lc
