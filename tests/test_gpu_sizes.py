"""Updates on graphs and batches whose sizes end at a tile, a warp or a block of
the kernels that sweep ids and sort batches, against the oracle: membership,
state and trace after every batch of a stream."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_2410_15451_gb300 import leiden as L
from paper_2410_15451_gb300 import synth

pytestmark = pytest.mark.gpu

MODES = [(L.LEIDEN_ND, oracle.ND), (L.LEIDEN_DS, oracle.DS), (L.LEIDEN_DF, oracle.DF)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2410_15451_gb300 import _build

    _build.build()
    L.load()


def same(gpu, ref):
    g, r = gpu.state(), ref.state()
    for k in ("C", "K", "Sigma", "dSigma"):
        assert np.array_equal(g[k], r[k]), k
    assert g["m2"] == r["m2"]
    assert gpu.trace() == ref.trace()
    for a, b in zip(gpu.graph(), ref.graph()):
        assert np.array_equal(a, b)


def sparse(n, seed):
    """Mean degree 3: many small communities, isolated vertices and pairs, so
    that communities appear, vanish and take freed ids."""
    return synth.planted_partition(n, max(1, n // 8), 3.0, 0.3, seed)


@pytest.mark.parametrize("mode", MODES, ids=["ND", "DS", "DF"])
@pytest.mark.parametrize("n", [2, 3, 33, 1023, 1024, 1025, 4097])
def test_ids_at_tile_edges(n, mode):
    g = sparse(n, 200 + n) if n > 8 else synth.Graph(n, np.array([0, 1, 2] + [2] * (n - 2), np.int64),
                                                     np.array([1, 0], np.int32), np.ones(2, np.int32))
    gpu = L.Leiden(g.n, g.off, g.col, g.w)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    assert np.array_equal(gpu.static(), ref.static())
    cur = g
    for k in range(4):
        size = max(1, n // 12) if n > 8 else 0
        if size:
            d, i = synth.random_batch(cur, size, seed=900 + k, frac_ins=[0.5, 0.1, 0.9, 0.3][k])
        else:  # the only edge goes and comes back
            e = np.array([[0, 1, 1]], np.int32)
            d, i = (e, e[:0]) if k % 2 == 0 else (e[:0], e)
        assert np.array_equal(gpu.update(d, i, mode[0]), ref.update(d, i, mode[1]))
        cur = synth.apply_batch_numpy(cur, d, i)
        same(gpu, ref)


@pytest.mark.parametrize("n_del,n_ins", [(0, 1), (1, 0), (0, 1024), (1, 1023), (512, 512), (1, 1024), (700, 325), (0, 0)])
def test_batches_at_the_one_block_limit(n_del, n_ins):
    """2 * (deletions + insertions) arcs up to 2048 are planned by one block, more
    by the sort's passes: repeated edges, insertions of existing edges, deleted
    edges inserted again and rows that outgrow their slack on both sides."""
    g = synth.planted_partition(3000, 30, 12.0, 0.2, 5)
    src = np.repeat(np.arange(g.n), np.diff(g.off))
    up = np.flatnonzero(src < g.col)
    rng = np.random.default_rng(n_del * 4099 + n_ins)
    for mode in MODES:
        gpu = L.Leiden(g.n, g.off, g.col, g.w, slack=0.0, min_slack=1)
        ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
        gpu.static(), ref.static()
        e = rng.choice(up, n_del, replace=n_del > 600)
        d = np.stack([src[e], g.col[e], np.ones(n_del, np.int64)], 1).astype(np.int32)
        u = rng.integers(0, g.n, n_ins)
        v = (u + rng.integers(1, g.n, n_ins)) % g.n
        i = np.stack([u, v, rng.integers(1, 5, n_ins)], 1).astype(np.int32)
        k = n_ins // 8
        again = rng.choice(up, k)  # existing edges, some of them deleted above
        i[:k, 0], i[:k, 1] = src[again], g.col[again]
        if n_del and k:
            i[0, :2] = d[0, 1], d[0, 0]
        i[k:2 * k, 0] = 7  # one row gets an eighth of the insertions
        i[:, 1] = np.where(i[:, 0] == i[:, 1], (i[:, 1] + 1) % g.n, i[:, 1])
        assert np.array_equal(gpu.update(d, i, mode[0]), ref.update(d, i, mode[1]))
        same(gpu, ref)


@pytest.mark.parametrize("size", [3, 1500])
def test_invalid_batches_leave_the_graph(size):
    """On both sides of the one-block limit: a bad edge among good ones."""
    g = synth.planted_partition(2000, 20, 10.0, 0.2, 62)
    gpu = L.Leiden(g.n, g.off, g.col, g.w)
    gpu.static()
    before = gpu.state()
    dels, ins = synth.random_batch(g, size, seed=4)
    absent = next(v for v in range(1, g.n) if v not in g.col[g.off[0]:g.off[1]])
    for d, i in [(np.vstack([dels, [[0, absent, 1]]]), ins), (dels, np.vstack([ins, [[3, 3, 1]]])),
                 (dels, np.vstack([ins, [[1, 2, 0]]])), (dels, np.vstack([ins, [[1, g.n, 1]]])),
                 (dels, np.vstack([ins, [[-1, 2, 1]]]))]:
        with pytest.raises(L.LeidenError) as e:
            gpu.update(d, i, L.LEIDEN_DF)
        assert e.value.status == L.LEIDEN_ERR_BATCH
        after = gpu.state()
        assert all(np.array_equal(before[k], after[k]) for k in ("C", "K", "Sigma", "dSigma"))
        assert np.array_equal(gpu.graph()[1], g.col)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    ref.static()
    assert np.array_equal(gpu.update(dels, ins, L.LEIDEN_DF), ref.update(dels, ins, oracle.DF))
    same(gpu, ref)


@pytest.mark.parametrize("arcs_each", [1, 8, 9, 40])
def test_rows_merged_at_every_class_limit(arcs_each):
    """Rows that end at a merge class's limit (256, 1024, 4096 arcs), with few and
    many batch arcs each, changed at the front, in the middle and at the end, in
    place and relocated."""
    lengths = [250, 256, 257, 1000, 1024, 1025, 4090, 4096, 4097, 5000]
    n = 6000
    hubs = {10 + 500 * k: m for k, m in enumerate(lengths)}
    edges = set()
    for h, m in hubs.items():
        others = [v for v in range(n) if v not in hubs][:m]
        edges |= {(min(h, v), max(h, v)) for v in others}
    from tests.helpers import csr_from_edges

    off, col, w = csr_from_edges(n, sorted(edges))
    rng = np.random.default_rng(arcs_each)
    for slack in (dict(slack=0.25, min_slack=64), dict(slack=0.0, min_slack=0)):
        gpu = L.Leiden(n, off, col, w.astype(np.int32), **slack)
        ref = oracle.Oracle(n, off, col, w.astype(np.int32), schedule=oracle.SYNC)
        gpu.static(), ref.static()
        d, i = [], []
        for h, m in hubs.items():
            row = col[off[h]:off[h + 1]]
            gone = [int(row[0]), int(row[-1])] + rng.choice(row, arcs_each).tolist()
            d += [(h, v, 1) for v in gone[:arcs_each]]
            there = set(row.tolist())
            absent = [v for v in range(n - 1, 0, -1) if v not in hubs and v not in there][:arcs_each]
            i += [(h, v, 2) for v in absent] + [(h, gone[0], 3)]  # one comes back with another weight
        for mode in MODES[2:]:
            assert np.array_equal(gpu.update(d, i, mode[0]), ref.update(d, i, mode[1]))
            same(gpu, ref)
            i2 = [(u, v, x) for u, v, x in i]
            assert np.array_equal(gpu.update(i2, [], mode[0]), ref.update(i2, [], mode[1]))  # all taken out again
            same(gpu, ref)


def check_stream(gpu, ref, g, steps, seed, modes=MODES, w_hi=1):
    """Random batches on both, state and trace compared after each."""
    cur = g
    for k in range(steps):
        mode = modes[k % len(modes)]
        d, i = synth.random_batch(cur, max(4, g.n // 100), seed=seed + k, frac_ins=[0.5, 0.2, 0.8][k % 3], w_lo=1, w_hi=w_hi)
        assert np.array_equal(gpu.update(d, i, mode[0]), ref.update(d, i, mode[1]))
        cur = synth.apply_batch_numpy(cur, d, i)
        same(gpu, ref)
    return cur


@pytest.mark.parametrize("classes", [1, 2, 16, 32, 64])
def test_any_number_of_classes(classes):
    """A local-moving iteration has a set of counters for 16 sub-sweeps, used again
    above that; with hubs (from 65 arcs on) and, as a batch, with two graphs."""
    gs = [synth.rmat(11, seed=31), synth.planted_partition(1500, 15, 10.0, 0.2, 32)]
    for g in gs:
        gpu = L.Leiden(g.n, g.off, g.col, g.w, classes=classes)
        L.leiden_set_tuning(gpu.h, tiny_max=4, warp_max=32, block_max=64)
        ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC, classes=classes)
        assert np.array_equal(gpu.static(), ref.static())
        same(gpu, ref)
        check_stream(gpu, ref, g, 3, 700)
    batch = L.LeidenBatch([(g.n, g.off, g.col, g.w) for g in gs], classes=classes)
    got = batch.static()
    for k, g in enumerate(gs):
        ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC, classes=classes)
        assert np.array_equal(batch.local(got, k), ref.static())


@pytest.mark.parametrize("block_max", [64, 1024])
def test_total_weight_passes_2_to_32_and_returns(block_max):
    """Sums by community are held in 32 bits while 2m is below 2^32: a handle that
    heavy insertions take above it and their deletion back, with random batches
    and a static call on either side; hubs and hub communities of both kinds."""
    g = synth.rmat(11, seed=44)
    gpu = L.Leiden(g.n, g.off, g.col, g.w)
    L.leiden_set_tuning(gpu.h, tiny_max=8, warp_max=64, block_max=block_max)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC)
    gpu.static(), ref.static()
    cur = check_stream(gpu, ref, g, 3, 400)
    for step, w in enumerate([(1 << 30) + 3, (1 << 30) + 3, 1 << 31 >> 1]):
        free = [(u, v) for u in range(5 * step, 5 * step + 3) for v in range(g.n - 1, 0, -1)
                if v > u and v not in set(cur.col[cur.off[u]:cur.off[u + 1]].tolist())][:3]
        heavy = np.array([(u, v, w) for u, v in free], np.int32)
        none = heavy[:0]
        assert np.array_equal(gpu.update(none, heavy, L.LEIDEN_DF), ref.update(none, heavy, oracle.DF))
        same(gpu, ref)
        assert gpu.state()["m2"] > 1 << 32
        cur = synth.apply_batch_numpy(cur, none, heavy)
        if step == 1:
            assert np.array_equal(gpu.static(), ref.static())
            same(gpu, ref)
        # (not of the heavy edges: they are deleted below)
        for k, mode in enumerate(MODES):
            edges = [(0, 100 + 7 * step + k, 2), (200, 300 + step, 1), (400 + k, 900, 5)]
            edges = np.array([e for e in edges if not any({e[0], e[1]} == {u, v} for u, v in free)], np.int32)
            assert np.array_equal(gpu.update(none, edges, mode[0]), ref.update(none, edges, mode[1]))
            cur = synth.apply_batch_numpy(cur, none, edges)
            same(gpu, ref)
        assert np.array_equal(gpu.update(heavy, none, MODES[step][0]), ref.update(heavy, none, MODES[step][1]))
        same(gpu, ref)
        assert gpu.state()["m2"] < 1 << 32
        cur = synth.apply_batch_numpy(cur, heavy, none)
        cur = check_stream(gpu, ref, cur, 3, 500 + 10 * step)
    assert np.array_equal(gpu.static(), ref.static())
    same(gpu, ref)


def spread(g, n):
    """g's vertices on ids spread evenly over [0, n), in order."""
    ids = (np.arange(g.n, dtype=np.int64) * n) // g.n
    deg = np.zeros(n, np.int64)
    deg[ids] = np.diff(g.off)
    return synth.Graph(n, np.concatenate([[0], np.cumsum(deg)]), ids[g.col].astype(np.int32), g.w)


@pytest.mark.parametrize("flags", [{}, dict(split_all=1)], ids=["changed", "all"])
def test_more_ids_than_one_tile_each(flags):
    """Above 2^21 vertices the split links in two steps, above 2^22 ids tracking's
    tiles take several steps: thin communities that deletions take apart, spread
    over 4,195,341 ids (an odd remainder), all other ids unused."""
    small = synth.planted_partition(20_000, 900, 5.0, 0.1, 77)
    g = spread(small, (1 << 22) + 1037)
    gpu = L.Leiden(g.n, g.off, g.col, g.w, **flags)
    ref = oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC, **flags)
    assert np.array_equal(gpu.static(), ref.static())
    same(gpu, ref)
    ids = (np.arange(small.n, dtype=np.int64) * g.n) // small.n
    for k, mode in enumerate(MODES):
        d, i = synth.random_batch(small, 2500, seed=60 + k, frac_ins=0.2)
        small = synth.apply_batch_numpy(small, d, i)
        d, i = [np.stack([ids[e[:, 0]], ids[e[:, 1]], e[:, 2]], 1).astype(np.int32) for e in (d, i)]
        assert np.array_equal(gpu.update(d, i, mode[0]), ref.update(d, i, mode[1]))
        same(gpu, ref)


def test_batch_of_graphs_with_more_ids_than_one_tile_each():
    """The second graph of a batch starts inside a tile of several steps."""
    parts = [synth.planted_partition(6000, 300, 5.0, 0.1, 78), synth.planted_partition(5000, 200, 5.0, 0.1, 79)]
    sizes = [(1 << 22) + 517, 70_001]
    gs = [spread(p, n) for p, n in zip(parts, sizes)]
    batch = L.LeidenBatch([(g.n, g.off, g.col, g.w) for g in gs])
    refs = [oracle.Oracle(g.n, g.off, g.col, g.w, schedule=oracle.SYNC) for g in gs]
    got = batch.static()
    for k, r in enumerate(refs):
        assert np.array_equal(batch.local(got, k), r.static())
    for step in range(2):
        dels, ins, want = [], [], []
        for k, r in enumerate(refs):
            d, i = synth.random_batch(parts[k], 900, seed=80 + 10 * step + k, frac_ins=0.3)
            parts[k] = synth.apply_batch_numpy(parts[k], d, i)
            ids = (np.arange(parts[k].n, dtype=np.int64) * sizes[k]) // parts[k].n
            d, i = [np.stack([ids[e[:, 0]], ids[e[:, 1]], e[:, 2]], 1).astype(np.int32) for e in (d, i)]
            want.append(r.update(d, i, oracle.DF))
            dels.append(batch.to_global(d, k))
            ins.append(batch.to_global(i, k))
        got = batch.update(np.concatenate(dels), np.concatenate(ins), L.LEIDEN_DF)
        for k, w in enumerate(want):
            assert np.array_equal(batch.local(got, k), w)
            for key in ("K", "Sigma", "dSigma"):
                a, b = int(batch.voff[k]), int(batch.voff[k + 1])
                assert np.array_equal(batch.state()[key][a:b], refs[k].state()[key])
