"""Requests submitted, polled and fetched on one thread while another one steps the
server (kb_server_submit is thread-safe with respect to kb_server_step), against
the oracle."""
import threading

import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402


@pytest.mark.parametrize("pinned", [True, False])
def test_submitted_while_stepping(pinned):
    graphs = [graphgen.erdos_renyi(n, 2 * n, 3, 2, seed=n) for n in (1, 50, 333, 2_000)]
    want = [oracle.refine_graph(g, kb.DIR_OUT, True, True, k=5) for g in graphs]

    def host(a):
        return torch.from_numpy(a.copy()).pin_memory().numpy() if pinned else a

    arrays = [[host(a) for a in (g.row_offsets, g.col, g.elabel, g.vlabel)] for g in graphs]
    bad, done = [], threading.Event()
    with kb.Server(0, max_vertices=1 << 16, max_edges=1 << 17, max_requests=32) as server:

        def client():
            try:
                tickets = []
                for i in range(2_000):
                    tickets.append((server.submit(*arrays[i % 4], 5), i % 4))
                    if len(tickets) < 40:
                        continue
                    for t, j in [x for x in tickets if server.poll(x[0]) == kb.Server.DONE]:
                        levels, counts, computed = server.fetch(t)
                        if not (np.array_equal(levels, want[j][0][:6]) and np.array_equal(counts, want[j][1])
                                and computed == want[j][2]):
                            bad.append(t)
                        tickets.remove((t, j))
                    server.stats()
                while tickets:
                    for t, j in [x for x in tickets if server.poll(x[0]) == kb.Server.DONE]:
                        if not np.array_equal(server.fetch(t)[0], want[j][0][:6]):
                            bad.append(t)
                        tickets.remove((t, j))
            except Exception as e:  # reported by the stepping thread
                bad.append(e)
            finally:
                done.set()

        thread = threading.Thread(target=client)
        thread.start()
        while not done.is_set():
            server.step()
        thread.join()
        assert not bad, bad[:3]
        stats = server.stats()
        assert stats["completed"] == stats["submitted"] == 2_000 and stats["running"] == stats["waiting"] == 0
