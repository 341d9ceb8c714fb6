"""Copies in and out that overlap the server's rounds, against the oracle: the
next request's arrays are copied while one is checked, rows of large requests
leave as soon as they are final, and a finished request's rows may still be on
their way when it is asked for."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

LARGE = 131_072  # rows of 512 KB


def request(n, seed, pinned):
    g = graphgen.erdos_renyi(n, 2 * n, 3, 2, seed=seed)

    def host(x):
        return torch.from_numpy(x.copy()).pin_memory().numpy() if pinned else x

    return g, [host(x) for x in (g.row_offsets, g.col, g.elabel, g.vlabel)]


@pytest.mark.parametrize("pinned", [False, True])
@pytest.mark.parametrize("d", [kb.DIR_OUT, kb.DIR_BOTH])
def test_rows_of_large_and_small_requests(pinned, d):
    sizes = [(LARGE, 6), (40, 2), (LARGE - 1, 3), (LARGE + 1, 9), (1, 4), (LARGE, 0), (LARGE, 1), (9_000, 12)]
    with kb.Server(0, max_vertices=1 << 20, max_edges=1 << 21, max_requests=5) as server:
        for rep in range(2):
            reqs = []
            for i, (n, k) in enumerate(sizes):
                g, host = request(n, 10 * rep + i, pinned)
                out = torch.full((k + 1, n), -7, dtype=torch.int32, pin_memory=pinned).numpy()
                opts = kb.Options(direction=d, early_stop=bool(i % 3))
                bad = i == 3 and rep == 0
                if bad:  # rejected while the one behind it is staged
                    host[1] = host[1].copy()
                    host[1][5] = n
                reqs.append((server.submit(*host, k, opts, out=out), g, k, out, opts, bad))
            left = list(reqs)
            stepped = True
            while left:
                if stepped:
                    server.step()
                stepped = True
                for r in left:
                    t, g, k, out, opts, bad = r
                    if server.poll(t) == 3:
                        assert bad
                        with pytest.raises(kb.KbError):
                            server.fetch(t)
                    elif server.poll(t) == 2:
                        L, C, lc = oracle.refine_graph(g, d, True, True, k=k, early_stop=opts.early_stop)
                        assert np.array_equal(out, L[:k + 1]), (g.n, k)  # before the fetch
                        levels, counts, computed = server.fetch(t)
                        assert levels is out and np.array_equal(counts, C) and computed == lc
                    else:
                        continue
                    left.remove(r)
                    stepped = False  # (a list that changed is walked again)
                    break
            assert server.stats()["running"] == 0


def test_closed_with_rows_on_their_way():
    server = kb.Server(0, max_vertices=1 << 20, max_edges=1 << 21, max_requests=4)
    out = torch.zeros((9, LARGE), dtype=torch.int32, pin_memory=True).numpy()
    g, host = request(LARGE, 5, True)
    server.submit(*host, 8, kb.Options(early_stop=False), out=out)
    server.submit(*request(LARGE, 6, True)[1], 1, kb.Options())
    for _ in range(3):
        server.step()
    server.close()
    L, _, _ = oracle.refine_graph(g, kb.DIR_OUT, True, True, k=2, early_stop=False)
    assert np.array_equal(out[:3], L)
