"""What a user of this library has it do, as measurable cases.

Every case is one call (or, for the server, one burst of requests) through the
public Python entry points: plain, prepared and host-buffer refinement, the
allocation-free round, full bisimulation, batches, serving, the summary graph
and incremental updates, over the graph families of the benchmark (power-law
graphs with Zipf labels, Erdos-Renyi graphs) and the trees of the tests.  The
graphs are drawn on the device from the seed.

Outputs are canonical block ids and counts, whole numbers without a rounding.
"""
import functools
import math

import numpy as np
import torch

import paper_2204_05821_gb300 as kb

DEVICE = "cuda:0"
MODELS = ("labelled", "schaetzle", "kaushik")
DIRECTIONS = {"out": kb.DIR_OUT, "in": kb.DIR_IN, "both": kb.DIR_BOTH}


def listed():
    return [
        # the smallest call: one summary of a toy graph, where launches and host round trips count
        dict(name="tiny er, out", call="refine", graph="er", n=10_000, m=50_000, vlabels=8, elabels=4,
             model="labelled", direction="out", k=10, early_stop=True),
        # one level at a time inside an application that may not allocate device memory
        dict(name="one round, no allocation", call="round", graph="er", n=100_003, m=480_017, vlabels=16, elabels=8,
             model="labelled", direction="out", k=1, early_stop=False),
        # a single summarisation request of median size, host arrays in and out
        dict(name="request from host memory", call="host", graph="power", n=140_000, m=700_000, gamma=2.1,
             vlabels=64, elabels=32, model="labelled", direction="out", k=5, early_stop=True),
        # a class hierarchy (child -> parent) refined until nothing changes: many small rounds
        dict(name="hierarchy to its fixpoint", call="fixpoint", graph="tree", n=300_007, m=300_006, vlabels=4,
             elabels=1, model="labelled", direction="out", k=200, early_stop=True),
        # a small edit of a finely labelled graph whose levels are known
        dict(name="update after an edit", call="update", graph="er", n=1_000_003, m=3_000_017, vlabels=200_000,
             elabels=3, model="labelled", direction="out", k=6, early_stop=True, changed=100),
        # backward bisimulation by vertex labels on an RDF-like graph, every level wanted
        dict(name="rdf, backward", call="refine", graph="power", n=1_000_000, m=10_000_000, gamma=2.1, vlabels=1000,
             elabels=200, model="kaushik", direction="in", k=10, early_stop=True),
        # forward and backward edges together, odd sizes, no early stop
        dict(name="rdf, both directions", call="refine", graph="power", n=2_500_003, m=25_000_019, gamma=2.1,
             vlabels=1000, elabels=200, model="labelled", direction="both", k=6, early_stop=False),
        # forward bisimulation by edge labels on the full-size RDF-like graph
        dict(name="rdf full size, forward", call="refine", graph="power", n=10_000_000, m=100_000_000, gamma=2.1,
             vlabels=1000, elabels=200, model="schaetzle", direction="out", k=10, early_stop=True),
        # the web-scale recipe at a tenth of its size, prepared once and refined again and again
        dict(name="large tenth, prepared", call="prepared", graph="power", n=20_000_000, m=200_000_000, gamma=2.0,
             vlabels=5000, elabels=500, model="labelled", direction="out", k=10, early_stop=True),
        # a layer of the summary graph, written out after a refinement
        dict(name="summary layer", call="summary", graph="power", n=2_000_000, m=20_000_000, gamma=2.1, vlabels=1000,
             elabels=200, model="labelled", direction="out", k=3, early_stop=True),
        # many independent graphs of uneven size in one call
        dict(name="batch of 512 graphs", call="batch", graph="er", graphs=512, median_m=50_000, vlabels=16, elabels=8,
             model="labelled", direction="out", k=10, early_stop=True),
        # a burst of requests to the server, host arrays in and out
        dict(name="burst of 16 requests", call="serve", graph="power", graphs=16, median_m=700_000, gamma=2.1,
             vlabels=64, elabels=32, model="labelled", direction="out", k=10, early_stop=True),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["refine", "refine", "refine", "prepared", "prepared", "host", "round", "fixpoint", "update",
                       "summary", "batch", "serve"])
    c = dict(call=call, k=rng.randint(2, 10), early_stop=rng.random() < 0.7)
    if call in ("batch", "serve"):
        if call == "batch":
            c.update(graph="er", graphs=_between(rng, 8, 600), median_m=_between(rng, 5_000, 60_000),
                     vlabels=rng.randint(2, 40), elabels=rng.randint(1, 12))
        else:
            c.update(graph="power", graphs=rng.randint(2, 20), median_m=_between(rng, 50_000, 800_000),
                     gamma=round(rng.uniform(2.0, 2.4), 2), vlabels=rng.randint(8, 100), elabels=rng.randint(4, 40))
        c.update(model="labelled", direction=rng.choice(["out", "out", "in", "both"]))
        return c
    c["model"] = rng.choice(MODELS)
    c["direction"] = {"schaetzle": "out", "kaushik": "in"}.get(c["model"]) or rng.choice(["out", "in", "both"])
    most_m = {"refine": 60_000_000, "prepared": 120_000_000, "host": 5_000_000, "round": 3_000_000,
              "fixpoint": 20_000_000, "update": 5_000_000, "summary": 25_000_000}[call]
    m = _between(rng, 20_000, most_m // 2 if c["direction"] == "both" else most_m)
    c.update(n=max(16, int(m / rng.uniform(3.0, 12.0))), m=m)
    if call == "round":
        c.update(n=min(c["n"], _round_limit()), graph="er", model="labelled", direction="out", k=1,
                 early_stop=False)
    elif call == "update":
        c.update(graph="er", changed=_between(rng, 5, 500))
    elif call == "fixpoint" and rng.random() < 0.6:
        n = _between(rng, 5_000, 3_000_000)
        c.update(graph="tree", n=n, m=n - 1, model="labelled", direction=rng.choice(["out", "in"]))
    else:
        c["graph"] = rng.choice(["power", "power", "power", "er"])
    if c["graph"] == "power":
        c.update(gamma=round(rng.uniform(2.0, 2.4), 2), vlabels=_between(rng, 8, 5000), elabels=_between(rng, 2, 500))
    elif call == "update":
        # labels fine enough that an edit touches a small part of the graph
        c.update(vlabels=max(2, c["n"] // rng.randint(3, 8)), elabels=rng.randint(1, 6))
    else:
        c.update(vlabels=rng.randint(2, 40), elabels=rng.randint(1, 12))
    if call == "fixpoint":
        c["k"] = 200
    return c


def _round_limit():
    """Vertices that the allocation-free round takes at most (KB_NOALLOC_MAX_VERTICES)."""
    return 1 << 20


# ----------------------------------------------------------------------------- graphs


def _generator(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _powerlaw_cdf(n, m, exponent, cap):
    """Cumulative capped Chung-Lu weights: rank r weighs r^(-1/(exponent-1)), at most `cap` expected edges."""
    d = torch.arange(1, n + 1, dtype=torch.float64, device=DEVICE).pow_(-1.0 / (exponent - 1.0))
    d *= m / d.sum()
    for _ in range(50):
        over = d > cap
        n_over = int(over.sum())
        if n_over == 0 or n_over == n:
            break
        d = torch.where(over, cap, d * ((m - cap * n_over) / d[~over].sum()))
    return _whole_cdf(d)


def _whole_cdf(weights):
    """Cumulative weights in whole numbers that sum to about 2^52: a parallel scan of them gives the same sums in
    whatever order it adds, so a seed always gives the same graph."""
    return (weights * (2.0 ** 52 / float(weights.sum()))).long().cumsum(0)


def _zipf_cdf(count, s):
    return _whole_cdf(torch.arange(1, max(1, count) + 1, dtype=torch.float64, device=DEVICE).pow_(-s))


def _draws(cdf, count, gen, chunk=1 << 26):
    """`count` draws of the distribution with this cumulative function, as int32."""
    out = torch.empty(count, dtype=torch.int32, device=DEVICE)
    total = int(cdf[-1])
    for a in range(0, count, chunk):
        b = min(count, a + chunk)
        u = torch.randint(0, total, (b - a,), device=DEVICE, generator=gen)
        out[a:b] = torch.searchsorted(cdf, u, right=True)
    return out


def _rows(deg):
    row = torch.zeros(deg.shape[0] + 1, dtype=torch.int64, device=DEVICE)
    torch.cumsum(deg, 0, out=row[1:])
    return row


def _uniform(count, below, gen):
    return torch.randint(0, max(1, below), (count,), dtype=torch.int32, device=DEVICE, generator=gen)


def _graph(kind, n, m, gamma, vlabels, elabels, gen):
    """(row_offsets, col, edge labels, vertex labels) of one graph on the device."""
    if kind == "power":
        # the recipes of the benchmark: hubs up to a tenth of the edges for small graphs, a thirtieth
        # (out) and a five-hundredth (in) for the web-scale one
        web = m >= 50_000_000
        cap_out, cap_in = (m / 30.0, m / 500.0) if web else (m / 10.0, m / 10.0)
        ranks = _draws(_powerlaw_cdf(n, m, gamma, cap_out), m, gen)
        deg = torch.empty(n, dtype=torch.int64, device=DEVICE)
        deg[torch.randperm(n, device=DEVICE, generator=gen)] = torch.bincount(ranks, minlength=n)
        del ranks
        col = _draws(_powerlaw_cdf(n, m, gamma, cap_in), m, gen)
        perm = torch.randperm(n, device=DEVICE, generator=gen).to(torch.int32)
        for a in range(0, m, 1 << 26):
            col[a:a + (1 << 26)] = perm[col[a:a + (1 << 26)]]
        return (_rows(deg), col, _draws(_zipf_cdf(elabels, 1.2), m, gen), _draws(_zipf_cdf(vlabels, 1.5), n, gen))
    if kind == "tree":
        # every vertex but the root has an edge to a parent drawn among the vertices before it
        ids = torch.randperm(n, device=DEVICE, generator=gen)
        later = torch.arange(1, n, device=DEVICE)
        u = torch.rand(n - 1, dtype=torch.float64, device=DEVICE, generator=gen)
        parent = torch.empty(n, dtype=torch.int32, device=DEVICE)
        parent[ids[1:]] = ids[(u * later).long().clamp_(max=n - 2)].to(torch.int32)
        deg = torch.ones(n, dtype=torch.int64, device=DEVICE)
        deg[ids[0]] = 0
        col = parent[torch.nonzero(deg).flatten()]
        return _rows(deg), col, _uniform(n - 1, elabels, gen), _uniform(n, vlabels, gen)
    deg = torch.bincount(torch.randint(0, n, (m,), device=DEVICE, generator=gen), minlength=n)
    return _rows(deg), _uniform(m, n, gen), _uniform(m, elabels, gen), _uniform(n, vlabels, gen)


def _sizes(case):
    """Edge counts of a batch or a burst: the quantiles of a lognormal distribution, the sizes in a fixed mixed
    order.  They are the case's; the seed draws only the graphs."""
    g = case["graphs"]
    sigma, lo, hi = (1.25, 1000, 2_000_000) if case["call"] == "batch" else (1.4, 10_000, 10_000_000)
    z = torch.special.ndtri((torch.arange(g, dtype=torch.float64) + 0.5) / g)
    ms = torch.exp(math.log(case["median_m"]) + sigma * z).clamp_(lo, hi).long()
    step = next(s for s in range(max(1, int(g * 0.618)), g + 2) if math.gcd(s, g) == 1)
    return [int(ms[(i * step) % g]) for i in range(g)], [1 + (i * 7) % case["k"] for i in range(g)]


def _options(case):
    kw = dict(early_stop=case["early_stop"])
    if case["model"] == "schaetzle":
        return kb.Options.schaetzle(**kw)
    if case["model"] == "kaushik":
        return kb.Options.kaushik(**kw)
    return kb.Options(direction=DIRECTIONS[case["direction"]], **kw)


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()


# ----------------------------------------------------------------------------- the calls


@functools.lru_cache(maxsize=None)
def _context():
    """The one context such a program keeps: its scratch serves every call."""
    return kb.Context(0)


def prepare(case, seed):
    gen = _generator(seed)
    s = dict(call=case["call"], k=case["k"], opts=_options(case), ctx=_context())
    if case["call"] == "batch":
        ms, ks = _sizes(case)
        ns = [max(1, m // 5) for m in ms]
        voff = np.concatenate([[0], np.cumsum(ns)]).astype(np.int64)
        n, m = int(voff[-1]), sum(ms)
        gid = torch.repeat_interleave(torch.arange(len(ms), device=DEVICE), torch.tensor(ms, device=DEVICE))
        first = torch.from_numpy(voff[:-1]).to(DEVICE)[gid]
        size = torch.tensor(ns, device=DEVICE)[gid]

        def ends():
            u = torch.rand(m, dtype=torch.float64, device=DEVICE, generator=gen)
            return first + torch.minimum((u * size).long(), size - 1)

        row = _rows(torch.bincount(ends(), minlength=n))
        # the edges of one graph are consecutive in the union, so the targets need no sorting
        s["graph"] = kb.DeviceGraph(row, ends().to(torch.int32), _uniform(m, case["elabels"], gen),
                                    _uniform(n, case["vlabels"], gen))
        s["voff"], s["ks"] = voff, np.asarray(ks, dtype=np.int32)
        return s
    if case["call"] == "serve":
        ms, ks = _sizes(case)
        s["requests"] = []
        for m, k in zip(ms, ks):
            host = [_pinned(t) for t in _graph(case["graph"], max(1, m // 5), m, case["gamma"], case["vlabels"],
                                               case["elabels"], gen)]
            out = torch.empty((k + 1, max(1, m // 5)), dtype=torch.int32, pin_memory=True).numpy()
            s["requests"].append((host, k, out))
        s["server"] = kb.Server(0, max_vertices=1 << 23, max_edges=1 << 26, max_requests=64)
        return s
    row, col, el, vl = _graph(case["graph"], case["n"], case["m"], case.get("gamma"), case["vlabels"],
                              case["elabels"], gen)
    if case["call"] == "host":
        s["host"] = [_pinned(t) for t in (row, col, el, vl)]
        s["out"] = torch.empty((case["k"] + 1, case["n"]), dtype=torch.int32, pin_memory=True).numpy()
        return s
    g = s["graph"] = kb.DeviceGraph(row, col, el, vl)
    if case["call"] == "prepared":
        s["graph"] = s["ctx"].prepare(g, s["opts"])
    elif case["call"] == "round":
        s["prev"] = s["ctx"].refine(g, 0, s["opts"]).levels[0]
        s["out"] = torch.empty_like(s["prev"])
    elif case["call"] == "summary":
        levels = s["ctx"].refine(g, case["k"], s["opts"]).levels
        s["src"], s["dst"] = levels[case["k"]].clone(), levels[case["k"] - 1].clone()
        s["direction"] = kb.DIR_IN if case["direction"] == "in" else kb.DIR_OUT
        s["layer"] = torch.zeros((3, case["m"]), dtype=torch.int32, device=DEVICE)
    elif case["call"] == "update":
        s["old"] = s["ctx"].refine(g, case["k"], s["opts"]).levels
        # the edit: some edges get another label
        edges = torch.randperm(case["m"], device=DEVICE, generator=gen)[:case["changed"]]
        new = el.clone()
        new[edges] = (new[edges] + 1) % (case["elabels"] + 1)
        sources = torch.searchsorted(row, edges, right=True) - 1
        ends = {"out": [sources], "in": [col[edges].long()], "both": [sources, col[edges].long()]}[case["direction"]]
        s["changed"] = torch.cat(ends).to(torch.int32)
        s["graph"] = kb.DeviceGraph(row, col, new, vl)
    return s


def run(s):
    ctx, call = s["ctx"], s["call"]
    if call in ("refine", "prepared"):
        r = ctx.refine(s["graph"], s["k"], s["opts"])
        return r.levels, r.counts, r.levels_computed
    if call == "host":
        r = ctx.refine_host(*s["host"], s["k"], s["opts"], out=s["out"])
        return r.levels, r.counts, r.levels_computed
    if call == "round":
        count = kb.refine_round_noalloc(s["graph"], s["prev"], s["out"], s["opts"])
        return s["out"], count
    if call == "fixpoint":
        return ctx.refine_fixpoint(s["graph"], s["k"], s["opts"])
    if call == "batch":
        return ctx.refine_batch(s["graph"], s["voff"], s["ks"], s["opts"])
    if call == "summary":
        # the layer goes to the head of the program's own arrays, which hold one entry per edge
        edges = ctx.summary(s["graph"], s["src"], s["dst"], direction=s["direction"])
        for own, part in zip(s["layer"], edges):
            own[:part.shape[0]] = part
        return s["layer"], edges[0].shape[0]
    if call == "update":
        # the levels are updated in place; the old ones are kept for the next edit
        r, work = ctx.refine_update(s["graph"], s["old"].clone(), s["changed"], s["opts"])
        return r.levels, r.counts, r.levels_computed, work
    server = s["server"]
    tickets = [server.submit(*host, k, s["opts"], out=out) for host, k, out in s["requests"]]
    while any(server.step()):
        pass
    done = [server.fetch(t) for t in tickets]
    return [d[0] for d in done], np.concatenate([d[1] for d in done]), np.asarray([d[2] for d in done])


def work(case):
    """Bytes of one call: the graph read once, the levels (or the summary's edges, at most one per edge) written once."""
    if case["call"] in ("batch", "serve"):
        ms, ks = _sizes(case)
        ns = [max(1, m // 5) for m in ms]
        rows = max(ks) + 1 if case["call"] == "batch" else None
        graph = sum(8 * (n + 1) + 4 * n + 8 * m for n, m in zip(ns, ms))
        return {"bytes": graph + sum(4 * n * (rows or k + 1) for n, k in zip(ns, ks)), "flops": 0}
    n, m, k = case["n"], case["m"], case["k"]
    elabel = 0 if case["model"] == "kaushik" else 4 * m
    vlabel = 0 if case["model"] == "schaetzle" else 4 * n
    graph = 8 * (n + 1) + 4 * m + elabel
    if case["call"] == "round":
        return {"bytes": graph + 4 * n + 4 * n, "flops": 0}
    if case["call"] == "summary":
        return {"bytes": 8 * (n + 1) + 8 * m + 8 * n, "flops": 0}
    if case["call"] == "fixpoint":
        return {"bytes": graph + vlabel + 4 * n, "flops": 0}
    if case["call"] == "update":
        return {"bytes": graph + vlabel + 8 * n * (k + 1), "flops": 0}
    return {"bytes": graph + vlabel + 4 * n * (k + 1), "flops": 0}
