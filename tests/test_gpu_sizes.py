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
