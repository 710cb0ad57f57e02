"""cvo_eval_gradient_static where most pairs are kept: launches of 8192 source points and
more then evaluate their work items in place instead of through the pair queue. The
sums are held to the FP64 oracle at ragged sizes, on both sides of the choice, with the
parity bars (F 1e-5, gradient 1e-4); coordinates that are no numbers or too large for
evaluation in place must leave the other pairs alone; and a call that keeps every pair must
not be the dearer kind: it evaluates 4e8 pairs where the other evaluates 5e6, about
2.2 times the time in place and 15 times through the queue."""
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


def _clouds(n, m, D, seed):
    rng = np.random.default_rng(seed)
    X = (rng.random((n, 3)) * 2 + [1.0, -2.0, 3.0]).astype(np.float32)
    Z = (rng.random((m, 3)) * 2 + [1.0, -2.0, 3.0]).astype(np.float32)
    return X, rng.random((n, D)).astype(np.float32), Z, rng.random((m, D)).astype(np.float32)


def _run(cvo, torch, X, FX, Z, FZ, P, ell, **kw):
    prm = cvo.cvo_params_default()
    for k, v in kw.items():
        setattr(prm, k, v)
    dev = [torch.from_numpy(a).cuda() for a in (X, FX, Z, FZ)]
    out = torch.full((8,), -1.0, dtype=torch.float64, device="cuda")
    cvo.cvo_eval_gradient_static(*dev, prm, P, ell, out)
    torch.cuda.synchronize()
    return out.cpu().numpy()


# kept: about 6% (queued), 25% and all of the pairs (in place)
@pytest.mark.parametrize("ell", [0.15, 0.26, 1.2])
@pytest.mark.parametrize("n,m,D,mode", [(5001, 8193, 5, 1), (4096, 8192, 3, 2), (2001, 15377, 8, 1),
                                        (6657, 8191, 0, 0), (33, 9000, 0, 0), (1, 8200, 5, 1)])
def test_dense_calls_match_the_oracle(cvo, n, m, D, mode, ell):
    torch = pytest.importorskip("torch")
    X, FX, Z, FZ = _clouds(n, m, max(D, 1), n + m)
    P = np.eye(4)
    P[:3, 3] = [0.01, -0.02, 0.005]
    got = [_run(cvo, torch, X, FX, Z, FZ, P, ell, feat_dim=D, color_mode=mode, color_scale=1.0)
           for _ in range(2)]
    assert np.array_equal(got[0], got[1])
    prm = oracle.Params(color_mode=mode, color_scale=1.0)
    ref = oracle.pair_sums(X, FX, Z, FZ, P, ell, prm)
    g = oracle.gradient(ref, prm)
    assert abs(got[0][0] - ref["F"]) <= 1e-5 * abs(ref["F"])
    assert np.linalg.norm(got[0][1:7] - g) <= 1e-4 * np.linalg.norm(g)
    assert abs(got[0][7] - ref["nnz"]) <= max(2, 1e-6 * ref["nnz"])


def test_wild_coordinates_keep_no_pair(cvo):
    """NaN, infinite and huge points among dense clouds: the sums are those without them.
    (Points are replaced, not removed, so that the tiles stay; FP32 sums in the same
    order up to the tiles that hold one: 1e-6.)"""
    torch = pytest.importorskip("torch")
    X, FX, Z, FZ = _clouds(6700, 8500, 5, 3)
    far = 1e9
    Xr, Zr = X.copy(), Z.copy()
    rows = {7: np.nan, 300: np.inf, 301: -np.inf, 4000: 3e38, 6699: 1e17}
    for i, v in rows.items():
        X[i, i % 3] = v
        Xr[i] = far
        Z[i % 8500, (i + 1) % 3] = v   # (not the same axis: two huge points could meet)
        Zr[i % 8500] = -far
    P = np.eye(4)
    got = _run(cvo, torch, X, FX, Z, FZ, P, 1.2)
    ref = _run(cvo, torch, Xr, FX, Zr, FZ, P, 1.2)
    assert np.isfinite(got).all()
    assert got[7] == ref[7] == (6700 - 5) * (8500 - 5)
    assert np.allclose(got[:7], ref[:7], rtol=0, atol=1e-6 * np.abs(ref[:7]).max())


def test_a_cutoff_beyond_every_number_keeps_all_pairs(cvo):
    torch = pytest.importorskip("torch")
    X, FX, Z, FZ = _clouds(6401, 8257, 1, 4)
    got = _run(cvo, torch, X, FX, Z, FZ, np.eye(4), 1e25, feat_dim=0, color_mode=0)
    assert got[7] == 6401 * 8257
    assert abs(got[0] - 6401 * 8257) <= 1e-6 * 6401 * 8257


def test_keeping_every_pair_is_not_the_dear_way(cvo):
    torch = pytest.importorskip("torch")
    n = 20000
    dev = [torch.from_numpy(a).cuda() for a in _clouds(n, n, 5, 5)]
    prm, P = cvo.cvo_params_default(), np.eye(4)
    out = torch.empty(8, dtype=torch.float64, device="cuda")
    ms = {}
    for ell in (0.08, 1.2):
        for _ in range(3):
            cvo.cvo_eval_gradient_static(*dev, prm, P, ell, out)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        for _ in range(10):
            cvo.cvo_eval_gradient_static(*dev, prm, P, ell, out)
        b.record()
        torch.cuda.synchronize()
        ms[ell] = a.elapsed_time(b) / 10
    assert ms[1.2] < 6.0 * ms[0.08], ms
