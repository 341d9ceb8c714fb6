"""A request that is fetched too early keeps its arrays and can be fetched later."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


def test_fetched_too_early():
    g = graphgen.path_graph(500)
    L, C, lc = oracle.refine_graph(g, kb.DIR_OUT, False, True, k=30)
    with kb.Server(0, max_vertices=1 << 12, max_edges=1 << 12, max_requests=2) as server:
        host = [a.copy() for a in (g.row_offsets, g.col, g.elabel, g.vlabel)]
        ticket = server.submit(*host, 30, kb.Options(use_vertex_labels=False))
        bad = host[1].copy()
        bad[3] = g.n
        rejected = server.submit(host[0], bad, host[2], host[3], 3)
        for step in range(3):  # waiting, then running
            with pytest.raises(kb.KbError):
                server.fetch(ticket)
            server.step()
        while any(server.step()):
            pass
        levels, counts, computed = server.fetch(ticket)
        assert np.array_equal(levels, L[:31]) and np.array_equal(counts, C) and computed == lc
        with pytest.raises(kb.KbError):
            server.fetch(rejected)
        for t in (ticket, rejected):  # forgotten
            with pytest.raises(KeyError):
                server.fetch(t)
