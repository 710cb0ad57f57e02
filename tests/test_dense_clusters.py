"""Clusters whose candidates all lie within the plan radius of their box go without the box test
of the streamed passes. The traversal's count of candidates shows it: with the test it
counts those that pass it, without it every point of the cells. A blob of 20000 points within
the cutoff of every source point, and points beside it that share a cell with points in reach
but are out of reach themselves: a few of them (no sample meets them) or many."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cvo():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1904_02266_gb300 as m
    return m


@pytest.mark.parametrize("beside,tested", [(0, False), (60, False), (9000, True)])
def test_dense_clusters_go_untested(cvo, beside, tested):
    rng = np.random.default_rng(8)
    m = 8003
    blob = rng.normal(scale=0.004, size=(20000, 3)).clip(-0.02, 0.02)
    out = rng.normal(scale=0.004, size=(beside, 3)).clip(-0.02, 0.02) + [0.455, 0.0, 0.0]
    X = np.concatenate([blob, out]).astype(np.float32)
    Z = rng.normal(scale=0.004, size=(m, 3)).clip(-0.02, 0.02).astype(np.float32)
    FX, FZ = rng.random((len(X), 5)).astype(np.float32), rng.random((m, 5)).astype(np.float32)
    P, ell = np.eye(4), 0.1          # cutoff 0.372, cells of 0.26
    with cvo.Context(device=0) as ctx:
        g = ctx.eval(ctx.set_cloud(X, FX), ctx.set_cloud(Z, FZ), P, ell)
    assert g["nnz"] == 20000 * m
    if tested:
        assert g["candidates"] < (20000 + beside // 2) * m
    else:
        assert g["candidates"] == len(X) * m
    ref = oracle.pair_sums(X, FX, Z, FZ, P, ell, oracle.Params())
    assert abs(g["F"] - ref["F"]) <= 1e-5 * ref["F"]
    gr = oracle.gradient(ref, oracle.Params())
    assert np.linalg.norm(g["grad6"] - gr) <= 1e-4 * np.linalg.norm(gr)
