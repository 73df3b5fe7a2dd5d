"""Kernels that walk rows by windows of 32 and cut long rows into chunks
(modularity, row sums, Delta-screening's neighbour expansion): rows of the
lengths where a window, a step or a chunk ends, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2410_15451_gb300 import leiden as L
from paper_2410_15451_gb300 import synth
from tests.helpers import csr_from_edges

pytestmark = pytest.mark.gpu

LENGTHS = {
    "short": [0, 1, 31, 32, 33, 0, 0, 127, 128, 129, 2, 0],
    "chunk": [4095, 4096, 4097, 0, 8191, 8193, 1, 0],
    "hub": [12289, 0, 5],
    "single": [1],
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_15451_gb300 import _build

    _build.build()
    L.load()


def stars(lengths, weighted):
    """Hubs spread over the ids, each joined to its own number of leaves (shared
    between the hubs), and isolated vertices at both ends."""
    leaves = max(lengths) if lengths else 0
    n = leaves + 3 * len(lengths) + 5
    hubs = [2 + 3 * k for k in range(len(lengths))]
    others = [v for v in range(2, n - 3) if v not in set(hubs)]
    edges = [(min(h, v), max(h, v)) for h, k in zip(hubs, lengths) for v in others[:k]]
    w = [(1 << 30) - 7 * i if weighted else 1 for i in range(len(edges))]
    off, col, wt = csr_from_edges(n, edges, w)
    return synth.Graph(n, off, col, wt.astype(np.int32))


@pytest.mark.parametrize("weighted", [False, True])
@pytest.mark.parametrize("name", sorted(LENGTHS))
def test_modularity_and_row_sums(name, weighted):
    import torch

    g = stars(LENGTHS[name], weighted)
    w64 = g.w.astype(np.int64)
    h = L.Leiden(g.n, g.off, g.col, g.w)
    d = [torch.from_numpy(x).cuda() for x in (g.off, g.col, g.w)]
    rng = np.random.default_rng(3)
    for C in (np.zeros(g.n, np.int32), np.arange(g.n, dtype=np.int32), rng.integers(0, min(7, g.n), g.n).astype(np.int32)):
        q, _ = oracle.modularity(g.off, g.col, w64, C)
        c = torch.from_numpy(C).cuda()
        assert h.modularity(C) == q
        assert L.leiden_modularity_noalloc(g.n, d[0], d[1], d[2], c) == q
        if not weighted:
            assert L.leiden_modularity_noalloc(g.n, d[0], d[1], None, c) == q
    h.static()
    st = h.state()
    K = np.zeros(g.n, np.int64)
    np.add.at(K, np.repeat(np.arange(g.n), np.diff(g.off)), w64)
    assert np.array_equal(st["K"], K) and st["m2"] == int(w64.sum())


@pytest.mark.parametrize("name", ["short", "chunk", "hub"])
def test_screening_expands_rows_of_every_length(name):
    g = stars(LENGTHS[name], False)
    gpu = L.Leiden(g.n, g.off, g.col, g.w)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    gpu.static(), ref.static()
    # an edge of every hub deleted (its row is expanded), edges between leaves and isolated vertices inserted
    dels = [(2 + 3 * k, int(g.col[g.off[2 + 3 * k]]), 1) for k in range(len(LENGTHS[name])) if LENGTHS[name][k]]
    ins = [(0, 3, 1), (1, 4, 2), (g.n - 1, 3, 1)]
    assert np.array_equal(gpu.update(dels, ins, L.LEIDEN_DS), ref.update(dels, ins, oracle.DS))
    assert np.array_equal(gpu.affected(), ref.affected())
    assert np.array_equal(gpu.state()["K"], ref.state()["K"])


HUB_SLOTS = [512, 513, 1025, 2048, 2049, 4097]  # distinct neighbour communities: warp, one piece, several pieces


@pytest.mark.parametrize("weighted", [False, True])
def test_hub_tables_of_every_size(weighted):
    """Hubs whose tables end at a warp's, a piece's and several pieces' limits,
    with 32-bit sums (unit weights) and with 64-bit ones (2m above 2^32); hubs
    that move mark their neighbours inline or in parts."""
    g = stars([max(k, 1030) if k < 1030 else k for k in HUB_SLOTS] + HUB_SLOTS, weighted)
    gpu = L.Leiden(g.n, g.off, g.col, g.w)
    L.leiden_set_tuning(gpu.h, block_max=256)  # the hub path from 257 arcs on
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    assert np.array_equal(gpu.static(), ref.static())
    assert gpu.trace() == ref.trace()
    dels = [(2 + 3 * k, int(g.col[g.off[2 + 3 * k]]), 1) for k in range(len(HUB_SLOTS))]
    assert np.array_equal(gpu.update(dels, [(0, 5, 1)], L.LEIDEN_ND), ref.update(dels, [(0, 5, 1)], oracle.ND))
    assert gpu.trace() == ref.trace()


def two_parts(n, part, degree, last):
    """Two rings of `part` vertices joined to their `degree` next ones, the first
    ids and the ids from `last` on; every other id is unused."""
    step = np.arange(1, degree // 2 + 1)
    v = np.arange(part)[:, None]
    row = np.sort(np.concatenate([(v + step) % part, (v - step) % part], 1), 1)
    off = np.zeros(n + 1, np.int64)
    off[1:part + 1] = degree
    off[last + 1:last + part + 1] = degree
    off = np.cumsum(off)
    col = np.concatenate([row.ravel(), row.ravel() + last]).astype(np.int32)
    return synth.Graph(n, off, col, np.ones(len(col), np.int32))


def fastest(call, runs=12):
    """Seconds of the quickest of `runs` calls that end with a wait for the GPU."""
    import time

    call()
    best = float("inf")
    for _ in range(runs):
        t = time.perf_counter()
        call()
        best = min(best, time.perf_counter() - t)
    return best


@pytest.mark.parametrize("unused", [31, 97, 160, 161, 4096, 1_000_000])
@pytest.mark.parametrize("part,degree", [(5, 2), (777, 30)])
def test_modularity_across_unused_ids(part, degree, unused):
    """A run of rows without arcs between two rows that have some."""
    import torch

    g = two_parts(2 * part + unused + 3, part, degree, part + unused)
    C = np.random.default_rng(unused).integers(0, 5, g.n).astype(np.int32)
    q, _ = oracle.modularity(g.off, g.col, g.w.astype(np.int64), C)
    d = [torch.from_numpy(x).cuda() for x in (g.off, g.col, g.w, C)]
    assert L.leiden_modularity_noalloc(g.n, d[0], d[1], d[2], d[3]) == q
    assert L.leiden_modularity_noalloc(g.n, d[0], d[1], None, d[3]) == q


def test_unused_ids_cost_no_more_in_the_middle_than_at_the_end():
    """One warp has the arcs on both sides of the run; at one step per 32 of its
    ids it would work for some 31,000 steps where the rest of the call has about
    ten (the bound leaves a factor of five for what else the call does)."""
    import torch

    part, unused = 20_001, 1_000_000  # (spans are multiples of 32 arcs: none ends between the parts)
    t = []
    for last in (part + unused, part):
        g = two_parts(2 * part + unused, part, 40, last)
        d = [torch.from_numpy(x).cuda() for x in (g.off, g.col, np.zeros(g.n, np.int32))]
        t.append(fastest(lambda: L.leiden_modularity_noalloc(g.n, d[0], d[1], None, d[2])))
    assert t[0] < 5 * t[1], t


def ring(n, degree, weighted=False):
    """Every vertex joined to the `degree` nearest ones of a ring."""
    g = two_parts(2 * n, n, degree, n)
    off, col = g.off[:n + 1].copy(), g.col[:n * degree].copy()
    src = np.repeat(np.arange(n), degree)
    w = 1 + (src + col) % 7 if weighted else np.ones(len(col))
    return synth.Graph(n, off, col, w.astype(np.int32))


@pytest.mark.parametrize("degree", [4, 6, 16, 32, 64, 130, 2048, 2050])
def test_windows_of_every_size(degree):
    """Mean degrees at which a small graph's windows have 32, 16, 8, 4 and 2 rows and a
    warp has one row (of up to 2048 arcs), the last window partly filled; one graph and two graphs whose boundary
    lies inside a window."""
    n = 3001
    g = ring(n, degree, True)
    w64 = g.w.astype(np.int64)
    K = np.add.reduceat(w64, g.off[:-1])
    C = np.random.default_rng(degree).integers(0, 9, n).astype(np.int32)
    q, _ = oracle.modularity(g.off, g.col, w64, C)
    h = L.Leiden(g.n, g.off, g.col, g.w)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    assert h.modularity(C) == q
    assert np.array_equal(h.static(), ref.static())
    assert np.array_equal(h.state()["K"], K)
    dels = [(5, 6, 1), (1500, 1501, 1), (0, n - 1, 1)]
    assert np.array_equal(h.update(dels, [(1, 1600, 3)], L.LEIDEN_DS), ref.update(dels, [(1, 1600, 3)], oracle.DS))
    assert np.array_equal(h.affected(), ref.affected())
    two = L.LeidenBatch([(g.n, g.off, g.col, g.w)] * 2)
    two.static()
    assert np.array_equal(two.state()["K"], np.concatenate([K, K]))
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    ref.static()
    assert list(two.modularity()) == [ref.modularity()] * 2


def test_a_small_dense_graph_fills_the_gpu():
    """Ten thousand rows of 2000 arcs: modularity on a handle (row sums first, two
    sweeps over the arcs) beside the call that cuts spans of arcs (one sweep).
    Windows of 32 rows would leave it to 313 of some 9,700 warps."""
    import torch

    g = ring(10_000, 2000)
    C = np.zeros(g.n, np.int32)
    d = [torch.from_numpy(x).cuda() for x in (g.off, g.col, g.w, C)]
    h = L.Leiden(g.n, g.off, g.col, g.w)
    t = fastest(lambda: h.modularity(C)), fastest(lambda: L.leiden_modularity_noalloc(g.n, d[0], d[1], d[2], d[3]))
    assert t[0] < 4 * t[1], t
