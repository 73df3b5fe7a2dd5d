"""What a user of the library has it do, as sized cases that can be timed.

A case is a dict of plain values.  ``prepare`` makes the inputs on the GPU from
a seed (graph, handle with its static clustering, a stream of batches),
``run`` is one call through the public entry points of
``paper_2410_15451_gb300.leiden``, ``work`` is the least a pass has to move,
and ``exact`` gives the floating-point outputs in 64 bits.

Kinds of case:

- ``static``: static Leiden of a resident graph.
- ``update``: one batch update of a tracked graph (ND, DS or DF).  The state
  holds a stream of distinct batches, 80% insertions of new edges and 20%
  deletions of original ones; passes apply them one after the other, and
  after the last one the stream is undone batch by batch (every insertion
  deleted, every deletion inserted again), so a state can be run for ever.
- ``rollback``: a large batch applied, the membership read, then the batch undone
  and the saved state imported again, so that every pass does the same work.
- ``batched``: updates as above, for many graphs in one handle.
- ``serve``: one update request for each graph of a server, all in flight at
  once, every membership waited for.
- ``modularity``: Q of a given membership on a caller-owned device CSR.

Memberships are whole numbers and the default (deterministic) schedule makes
them the same on every run.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2410_15451_gb300 import leiden as L

MODES = {"ND": L.LEIDEN_ND, "DS": L.LEIDEN_DS, "DF": L.LEIDEN_DF}


def listed():
    return [
        # A small network clustered from scratch and its state saved (the small
        # configuration: 10,000 vertices in blocks of 100, mean degree 16, mixing 0.2):
        # several passes over a graph that fits in a few SMs, so launches and host
        # round trips count.
        dict(name="static_planted_10k", kind="static", graph="planted", n=10_000, degree=16.0, state=True),
        # The small configuration's update: 100 edges, host arrays in, membership out.
        dict(name="df_planted_10k", kind="update", graph="planted", n=10_000, degree=16.0, mode="DF", batch=100,
             stream=32, device=False),
        # An event stream on a mid-sized social-network-like graph (R-MAT): a handful of
        # edges per update, the smallest batches that the service takes; an odd vertex count.
        dict(name="df_rmat20_16_edges", kind="update", graph="rmat", n=1_000_003, degree=32.0, mode="DF", batch=16,
             stream=1024, device=True),
        # The main configuration: R-MAT scale 22, batches of 1e-3 of its edges, on the device.
        dict(name="df_rmat22_1e-3", kind="update", graph="rmat", n=1 << 22, degree=32.0, mode="DF", batch=64_154,
             stream=160, device=True),
        # The two other markings, at 1e-3 of the edges of a quarter-size graph, through the
        # host arrays of the Python class.
        dict(name="nd_rmat20_1e-3", kind="update", graph="rmat", n=1 << 20, degree=32.0, mode="ND", batch=15_700,
             stream=192, device=False),
        dict(name="ds_rmat20_1e-3", kind="update", graph="rmat", n=1 << 20, degree=32.0, mode="DS", batch=15_700,
             stream=192, device=False),
        # The largest batches of the sweep, 0.1 of the edges at once, as a what-if: applied, read,
        # and taken back to the saved state.  Many passes and iterations.
        dict(name="rollback_rmat20_0.1", kind="rollback", graph="rmat", n=1 << 20, degree=32.0, mode="DF",
             batch=1_570_000),
        # The first clustering of a large resident graph.
        dict(name="static_rmat21", kind="static", graph="rmat", n=1 << 21, degree=32.0, state=False),
        # A web-like graph: power-law degrees and community sizes, weights 1..8, ragged
        # sizes, batches of 1e-4 of its edges.
        dict(name="df_web_1e-4", kind="update", graph="web", n=777_777, degree=50.0, mode="DF", batch=1_900, stream=128,
             device=True),
        # Many small graphs of uneven size in one handle, each with 1e-3 of its edges.
        dict(name="df_batched_96", kind="batched", graphs=96, n_lo=1_000, n_hi=50_000, deg_lo=4.0, deg_hi=64.0,
             fraction=1e-3, stream=64),
        # Serving: a request of its own size for each of eight resident graphs, four slots.
        dict(name="serve_8_graphs", kind="serve", graphs=8, scale_lo=15, scale_hi=18, batch_lo=10, batch_hi=3_000,
             slots=4, stream=48),
        # Quality of a clustering on a caller's own arrays, without allocation.
        dict(name="modularity_rmat22", kind="modularity", graph="rmat", n=1 << 22, degree=32.0, communities=20_000,
             weighted=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["static", "update", "update", "update", "update", "batched", "serve", "modularity"])
    if kind == "batched":
        lo = int(_log(rng, 500, 5_000))
        return dict(kind=kind, graphs=rng.randint(2, 120), n_lo=lo, n_hi=int(lo * rng.uniform(2, 10)), deg_lo=4.0,
                    deg_hi=round(rng.uniform(8, 64), 1), fraction=round(_log(rng, 3e-4, 3e-3), 6), stream=64)
    if kind == "serve":
        lo = rng.randint(12, 16)
        return dict(kind=kind, graphs=rng.randint(2, 12), scale_lo=lo, scale_hi=lo + rng.randint(0, 18 - lo), batch_lo=10,
                    batch_hi=int(_log(rng, 100, 3_000)), slots=rng.randint(1, 6), stream=48)
    graph = rng.choice(["planted", "rmat", "web"])
    n = int(_log(rng, 3_000, 1_500_000))
    degree = round(_log(rng, 6, 48), 1)
    if kind == "static":
        return dict(kind=kind, graph=graph, n=n, degree=degree, state=rng.random() < 0.3)
    if kind == "modularity":
        return dict(kind=kind, graph=graph, n=n, degree=degree, communities=max(16, int(n / _log(rng, 10, 10_000))),
                    weighted=rng.random() < 0.5)
    if rng.random() < 0.2:
        return dict(kind="rollback", graph=graph, n=min(n, 1_000_000), degree=min(degree, 32.0),
                    mode=rng.choice(["ND", "DS", "DF"]),
                    batch=int(min(n, 1_000_000) * min(degree, 32.0) / 2 * rng.uniform(0.01, 0.1)))
    batch = max(1, int(n * degree / 2 * _log(rng, 1e-6, 0.01)))
    return dict(kind=kind, graph=graph, n=n, degree=degree, mode=rng.choice(["ND", "DS", "DF", "DF"]), batch=batch,
                stream=max(2, min(128, int(0.3 * n * degree / 2 / batch))), device=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs
def _rand(k, gen):
    return torch.rand(k, generator=gen, device="cuda", dtype=torch.float32)


def _ints(hi, k, gen):
    return torch.randint(0, hi, (k,), generator=gen, device="cuda", dtype=torch.int64)


def _power_law(k, exponent, lo, hi, gen):
    """k draws of density ~ x^-exponent in [lo, hi] (64-bit)."""
    u = torch.rand(k, generator=gen, device="cuda", dtype=torch.float64)
    e = 1.0 - exponent
    return (lo ** e + u * (hi ** e - lo ** e)) ** (1.0 / e)


def _pairs_rmat(n, m, gen):
    """R-MAT pairs (a=0.57, b=c=0.19, d=0.05) on randomly permuted ids."""
    scale = max(1, (n - 1).bit_length())
    u = torch.zeros(m, dtype=torch.int64, device="cuda")
    v = torch.zeros(m, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = _rand(m, gen)
        u = u * 2 + (r >= 0.76)
        v = v * 2 + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    perm = torch.randperm(1 << scale, generator=gen, device="cuda")
    return perm[u] % n, perm[v] % n


def _pairs_planted(n, m, gen, block=100, mixing=0.2):
    """Consecutive blocks of `block` vertices, a share `mixing` of the pairs across them."""
    u = _ints(n, m, gen)
    inside = torch.minimum((u // block) * block + _ints(block, m, gen), torch.tensor(n - 1, device="cuda"))
    return u, torch.where(_rand(m, gen) < mixing, _ints(n, m, gen), inside)


def _pairs_web(n, m, gen, mixing=0.3):
    """Degree-corrected planted partition: power-law expected degrees (exponent 2.1) and
    community sizes (exponent 1.5, from 10 up), a share `mixing` across communities."""
    deg = _power_law(n, 2.1, 1.0, max(2.0, n / 50.0), gen)
    sizes = _power_law(max(1, n // 10), 1.5, 10.0, max(20.0, n / 30.0), gen).long()
    ends = torch.cumsum(sizes, 0).clamp(max=n)
    cum = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), torch.cumsum(deg, 0)])
    perm = torch.randperm(n, generator=gen, device="cuda")

    def at(x):  # the vertex whose share of the total degree holds x
        return (torch.searchsorted(cum, x, right=True) - 1).clamp(0, n - 1)

    u = at(torch.rand(m, generator=gen, device="cuda", dtype=torch.float64) * cum[-1])
    k = torch.searchsorted(ends, u, right=True).clamp(max=len(ends) - 1)
    lo = cum[torch.where(k > 0, ends[k - 1], torch.zeros_like(k))]
    hi = cum[ends[k]]
    r = torch.rand(m, generator=gen, device="cuda", dtype=torch.float64)
    v = torch.where(_rand(m, gen) < mixing, at(r * cum[-1]), at(lo + r * (hi - lo)))
    return perm[u], perm[v]


PAIRS = {"rmat": _pairs_rmat, "planted": _pairs_planted, "web": _pairs_web}


def _edges(graph, n, degree, gen):
    """Distinct undirected edges as sorted keys lo * n + hi, and their weights (None = unit)."""
    u, v = PAIRS[graph](n, max(1, int(n * degree / 2)), gen)
    keep = u != v
    u, v = u[keep], v[keep]
    key = torch.unique(torch.minimum(u, v) * n + torch.maximum(u, v))
    w = (1 + _ints(8, len(key), gen)).int() if graph == "web" else None
    return key, w


def _csr(n, key, w):
    """Symmetric CSR of the edges on the GPU: off int64, col int32, w int32 or None; rows sorted."""
    lo, hi = key // n, key % n
    arc, order = torch.sort(torch.cat([key, hi * n + lo]))
    src = arc // n
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return off, (arc % n).int(), None if w is None else torch.cat([w, w])[order]


def _stream(n, key, w, batch, stream, gen):
    """`stream` batches as (deletions, insertions), int32 (k, 3) tensors on the GPU: edges of
    the graph to delete and pairs that are no edges to insert, none of them twice."""
    n_ins = batch - int(round(0.2 * batch))
    n_del = min(batch - n_ins, len(key) // (2 * stream))
    new = torch.zeros(0, dtype=torch.int64, device="cuda")
    want = min(n_ins * stream, n * (n - 1) // 4)
    while len(new) < want:
        k = want + want // 8 + 64
        a, b = _ints(n, k, gen), _ints(n, k, gen)
        new = torch.unique(torch.cat([new, (torch.minimum(a, b) * n + torch.maximum(a, b))[a != b]]))
        at = torch.searchsorted(key, new).clamp(max=len(key) - 1)
        new = new[key[at] != new]
    new = new[torch.randperm(len(new), generator=gen, device="cuda")]
    old = torch.randperm(len(key), generator=gen, device="cuda")[: n_del * stream]
    new_w = (1 + _ints(8, len(new), gen)) if w is not None else torch.ones_like(new)
    old_w = w[old] if w is not None else torch.ones_like(old)

    def triples(k, x):
        return torch.stack([k // n, k % n, x.long()], 1).int().contiguous()

    dels, ins = triples(key[old], old_w), triples(new, new_w)
    n_ins = min(n_ins, len(new) // stream)
    return [(dels[i * n_del:(i + 1) * n_del], ins[i * n_ins:(i + 1) * n_ins]) for i in range(stream)]


def _spread(i, step, lo, hi):
    """The i-th of sizes that fill [lo, hi] evenly over their logarithm (the same for every seed)."""
    return lo * (hi / lo) ** ((0.5 + i * step) % 1.0)


def _host(x):
    return None if x is None else x.cpu().numpy()


def _graph(case, gen):
    key, w = _edges(case["graph"], case["n"], case["degree"], gen)
    return key, w, _csr(case["n"], key, w)


def _there_and_back(batches, at):
    """Batch number `at` of the endless stream: all of them forwards, then undone backwards."""
    k = at % (2 * len(batches))
    if k < len(batches):
        return batches[k]
    d, i = batches[2 * len(batches) - 1 - k]
    return i, d


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    kind = case["kind"]
    state = {"case": dict(case), "at": 0}
    if kind in ("static", "update", "rollback"):
        n = case["n"]
        key, w, (off, col, wt) = _graph(case, gen)
        state["h"] = L.Leiden(n, _host(off), _host(col), _host(wt))
        if kind == "update":
            batches = _stream(n, key, w, case["batch"], case["stream"], gen)
            if case["device"]:
                state["out"] = torch.zeros(n, dtype=torch.int32, device="cuda")
            else:
                batches = [(_host(d), _host(i)) for d, i in batches]
            state["batches"] = batches
            L.leiden_static(state["h"].h)
        if kind == "rollback":
            (dels, ins), = _stream(n, key, w, case["batch"], 1, gen)
            state.update(dels=_host(dels), ins=_host(ins))
            L.leiden_static(state["h"].h)
            state["saved"] = state["h"].state()
    elif kind == "batched":
        graphs, streams = [], []
        for i in range(case["graphs"]):
            n = int(_spread(i, 0.618034, case["n_lo"], case["n_hi"]))
            key, w = _edges("planted", n, min(_spread(i, 0.754878, case["deg_lo"], case["deg_hi"]), 40.0), gen)
            off, col, _ = _csr(n, key, w)
            graphs.append((n, _host(off), _host(col), None))
            streams.append([(_host(d), _host(i)) for d, i in _stream(
                n, key, w, max(1, int(len(key) * case["fraction"])), case["stream"], gen)])
        state["h"] = L.LeidenBatch(graphs)
        state["batches"] = [
            tuple(np.concatenate([state["h"].to_global(s[k][part], i) for i, s in enumerate(streams)]) for part in (0, 1))
            for k in range(case["stream"])]
        state["h"].static()
    elif kind == "serve":
        server = L.LeidenServer(60 << 30, slots=case["slots"])
        state["server"], state["graphs"] = server, []
        for i in range(case["graphs"]):
            n = 1 << (case["scale_lo"] + i % (case["scale_hi"] - case["scale_lo"] + 1))
            key, w = _edges("rmat", n, 32.0, gen)
            off, col, _ = _csr(n, key, w)
            batch = int(_spread(i, 0.618034, case["batch_lo"], case["batch_hi"]))
            batches = [(_host(d), _host(i)) for d, i in _stream(n, key, w, batch, case["stream"], gen)]
            state["graphs"].append((server.add_graph(n, _host(off), _host(col)), batches))
        for g, _ in state["graphs"]:
            server.membership(g)  # resident and clustered
    else:
        n = case["n"]
        key, w, (off, col, wt) = _graph(case, gen)
        if case["weighted"] and wt is None:
            w = (1 + _ints(8, len(key), gen)).int()
            off, col, wt = _csr(n, key, w)
        elif not case["weighted"]:
            wt = None
        # a rough clustering: ids in runs of vertices, a tenth of the vertices elsewhere
        c = torch.arange(n, device="cuda") * case["communities"] // n
        c = torch.where(_rand(n, gen) < 0.1, _ints(case["communities"], n, gen), c)
        state.update(off=off, col=col, w=wt, C=c.int())
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    at = state["at"]
    state["at"] = at + 1
    if kind == "static":
        c = state["h"].static()
        return {"membership": c, **state["h"].state()} if case["state"] else {"membership": c}
    if kind == "update":
        dels, ins = _there_and_back(state["batches"], at)
        if case["device"]:
            L.leiden_update_device(state["h"].h, dels, len(dels), ins, len(ins), MODES[case["mode"]], state["out"])
            return {"membership": state["out"]}
        return {"membership": state["h"].update(dels, ins, MODES[case["mode"]])}
    if kind == "rollback":
        h, mode = state["h"], MODES[case["mode"]]
        c = h.update(state["dels"], state["ins"], mode)
        undone = h.update(state["ins"], state["dels"], mode)
        L.leiden_import_state(h.h, state["saved"]["C"], state["saved"]["dSigma"])
        return {"membership": c, "undone": undone}
    if kind == "batched":
        dels, ins = _there_and_back(state["batches"], at)
        return {"membership": state["h"].update(dels, ins, L.LEIDEN_DF)}
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(g, *_there_and_back(batches, at), L.LEIDEN_DF, keep_membership=True)
                   for g, batches in state["graphs"]]
        return {"memberships": [server.wait(t)[0] for t in tickets]}
    q = L.leiden_modularity_noalloc(case["n"], state["off"], state["col"], state["w"], state["C"])
    return {"q": q}


def work(case):
    """The least a pass moves: the arcs that have to be looked at (column, weight and the
    neighbour's community, 12 B), the batch (12 B an edge), the membership read and written."""
    kind = case["kind"]
    if kind == "batched":
        n = case["graphs"] * (case["n_hi"] - case["n_lo"]) / math.log(case["n_hi"] / case["n_lo"])
        degree = (case["deg_hi"] - case["deg_lo"]) / math.log(case["deg_hi"] / case["deg_lo"])
        batch = n * degree / 2 * case["fraction"]
    elif kind == "serve":
        scales = range(case["scale_lo"], case["scale_hi"] + 1)
        n = case["graphs"] * sum(1 << s for s in scales) / len(scales)
        degree = 32.0
        batch = case["graphs"] * (case["batch_hi"] - case["batch_lo"]) / math.log(case["batch_hi"] / case["batch_lo"])
    else:
        n, degree, batch = case["n"], case["degree"], case.get("batch", 0)
    if kind == "static":
        return {"bytes": 12 * n * degree + (12 + 8) * n + (24 * n if case["state"] else 0), "flops": 0}
    if kind == "modularity":
        return {"bytes": (12 if case["weighted"] else 8) * n * degree + 12 * n, "flops": 0}
    # the rows that the batch touches (twice its edges at most, every row for ND) are read once
    rows = n if case.get("mode") == "ND" else min(n, 2 * batch)
    times = 2 if kind == "rollback" else 1
    return {"bytes": times * (12 * batch + 12 * rows * degree + 8 * n), "flops": 0}


def exact(case, seed):
    """Q in 64 bits, Eq. 1: intra-community weight over 2m, less the squared community shares."""
    if case["kind"] != "modularity":
        return None
    s = prepare(case, seed)
    n = case["n"]
    off, c = s["off"], s["C"].long()
    src = torch.repeat_interleave(torch.arange(n, device="cuda"), off[1:] - off[:-1])
    w = torch.ones(len(src), dtype=torch.float64, device="cuda") if s["w"] is None else s["w"].double()
    m2 = w.sum()
    inside = (w * (c[src] == c[s["col"].long()])).sum()
    sigma = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, c[src], w)
    return {"q": float(inside / m2 - ((sigma / m2) ** 2).sum())}
