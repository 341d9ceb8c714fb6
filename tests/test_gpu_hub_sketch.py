"""Hub sketches (csrc/kb_hub.cu), against the oracle: hubs that are alone, hubs
whose pair sets are equal although their edges repeat and are ordered
differently, and hubs with so few distinct pairs that small and medium vertices
share their signature."""
import numpy as np
import pytest

import graphgen
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_2204_05821_gb300 as kb  # noqa: E402

N, TARGETS = 30_000, 20_000


@pytest.fixture(scope="module")
def ctx():
    c = kb.Context(0)
    yield c
    c.close()


def hub_graph(seed, labels):
    """Vertices below TARGETS are what hubs point to (most with edges of their own, so that their blocks split)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lists = {}  # vertex -> (targets, labels)
    hub = TARGETS
    for size in (1500, 2500, 9000, 40_000):
        for twins in (1, 1, 2, 3):
            base = rng.choice(TARGETS, size=min(size, 15_000), replace=False)
            lab = rng.integers(0, labels, size=base.shape[0])
            for _ in range(twins):  # the same distinct edges, repeated and shuffled differently
                extra = rng.integers(0, base.shape[0], size=size // 3 + int(rng.integers(0, 500)))
                order = rng.permutation(np.concatenate([np.arange(base.shape[0]), extra]))
                lists[hub] = (base[order], lab[order])
                hub += 1
    for distinct in (1, 3, 20, 100, 900):  # few distinct edges: shared with vertices of every degree class
        base = rng.choice(TARGETS, size=distinct, replace=False)
        lab = rng.integers(0, labels, size=distinct)
        for size in (distinct, 2 * distinct + 1, 60, 400, 2000, 5000):
            order = rng.permutation(np.concatenate([np.arange(distinct), rng.integers(0, distinct, size=max(0, size - distinct))]))
            lists[hub] = (base[order], lab[order])
            hub += 1
    src = [np.full(t.shape[0], v) for v, (t, _) in lists.items()]
    dst = [t for t, _ in lists.values()]
    lab = [l for _, l in lists.values()]
    filler = 3 * TARGETS
    src.append(rng.integers(0, TARGETS, size=filler))
    dst.append(rng.integers(0, N, size=filler))
    lab.append(rng.integers(0, labels, size=filler))
    # a million edges between further unique hubs and the targets, so that there are enough chunks
    for v in range(hub, hub + 90):
        src.append(np.full(12_000, v))
        dst.append(rng.integers(0, TARGETS, size=12_000))
        lab.append(rng.integers(0, labels, size=12_000))
    vl = rng.integers(0, 3, size=N)
    vl[TARGETS:] = 0  # hubs start in one block
    return graphgen.from_edges(N, np.concatenate(src), np.concatenate(dst), np.concatenate(lab), vl)


@pytest.fixture(scope="module")
def graphs():
    return [hub_graph(1, 3), hub_graph(2, 1)]


def compare(res, g, d, k, opts):
    L, C, lc = oracle.refine_graph(g, d, opts.use_vertex_labels, opts.use_edge_labels, k=k, early_stop=opts.early_stop)
    got = res.levels.cpu().numpy()
    for i in range(k + 1):
        assert np.array_equal(got[i], L[i]), (d, opts, "level %d" % i)
    assert np.array_equal(res.counts, C) and res.levels_computed == lc


@pytest.mark.parametrize("kw", [dict(), dict(rekey_all=True), dict(hash_mode=1), dict(hub_threshold=128),
                                dict(hub_threshold=127), dict(hub_chunk_edges=256), dict(hub_chunk_edges=1024),
                                dict(use_vertex_labels=False), dict(use_edge_labels=False)])
def test_sketches_leave_every_level(ctx, graphs, kw):
    for g in graphs:
        dg = kb.DeviceGraph.from_numpy(g, "cuda:0")
        for d in (kb.DIR_OUT, kb.DIR_BOTH):
            opts = kb.Options(direction=d, early_stop=False, **kw)
            compare(ctx.refine(dg, 4, opts), g, d, 4, opts)
            opts = kb.Options(direction=d, reorder=2, **kw)
            with ctx.prepare(dg, opts) as pg:
                compare(ctx.refine(pg, 4), g, d, 4, opts)


def test_sketches_in_batches_and_updates(ctx, graphs):
    union, voff = graphgen.disjoint_union(graphs + [graphgen.make(graphgen.CONFIG_TINY)])
    levels, counts, lc = ctx.refine_batch(kb.DeviceGraph.from_numpy(union, "cuda:0"), voff, [3, 4, 2], kb.Options())
    levels = levels.cpu().numpy()
    for j, (g, k) in enumerate(zip(graphs, (3, 4))):
        L, C, last = oracle.refine_graph(g, 0, True, True, k=k)
        for i in range(5):
            assert np.array_equal(levels[i, voff[j]:voff[j + 1]], L[min(i, k)]), (j, i)
        assert lc[j] == last
    g = graphs[0]
    old = ctx.refine(kb.DeviceGraph.from_numpy(g, "cuda:0"), 4, kb.Options()).levels.clone()
    el = g.elabel.copy()
    e = int(g.row_offsets[TARGETS + 5])  # an edge of a hub with a twin
    el[e] += 1
    g2 = graphgen.Graph(n=g.n, m=g.m, row_offsets=g.row_offsets, col=g.col, elabel=el, vlabel=g.vlabel)
    changed = torch.tensor([TARGETS + 5], dtype=torch.int32, device="cuda:0")
    res, _ = ctx.refine_update(kb.DeviceGraph.from_numpy(g2, "cuda:0"), old, changed, kb.Options())
    compare(res, g2, 0, 4, kb.Options())
