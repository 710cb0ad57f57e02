"""cvo_eval_gradient_static at the edges of its tiles (256 source points, up to
256 targets tested 32 at a time) and of its pair queue (no pair, a few, every
pair kept), against the FP64 oracle. Tolerances are the parity bars: F 1e-5,
gradient 1e-4; the kept pairs may differ by those within rounding of the cutoff."""
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


@pytest.mark.parametrize("spread", [0.02, 0.4, 2.0])   # every pair kept, some, few
@pytest.mark.parametrize("n,m", [(1, 1), (31, 65), (32, 64), (33, 255), (255, 256), (257, 257),
                                 (513, 33), (1021, 1543), (4099, 7001)])
def test_tile_edges(cvo, n, m, spread):
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(n * 31 + m)
    X = (rng.normal(scale=spread, size=(n, 3)) + [1.0, -2.0, 3.0]).astype(np.float32)
    Z = (X[rng.integers(0, n, m)] + rng.normal(scale=0.02, size=(m, 3))).astype(np.float32)
    FX, FZ = rng.random((n, 5)).astype(np.float32), rng.random((m, 5)).astype(np.float32)
    P = np.eye(4)
    P[:3, 3] = [0.01, -0.02, 0.005]
    params, prm = cvo.cvo_params_default(), oracle.Params()
    out = torch.full((8,), -1.0, dtype=torch.float64, device="cuda")
    dev = [torch.from_numpy(a).cuda() for a in (X, FX, Z, FZ)]
    got = []
    for _ in range(2):
        cvo.cvo_eval_gradient_static(*dev, params, P, 0.15, out)
        torch.cuda.synchronize()
        got.append(out.cpu().numpy().copy())
    assert np.array_equal(got[0], got[1])
    ref = oracle.pair_sums(X, FX, Z, FZ, P, 0.15, prm)
    g = oracle.gradient(ref, prm)
    assert abs(got[0][0] - ref["F"]) <= 1e-5 * ref["F"]
    assert np.linalg.norm(got[0][1:7] - g) <= 1e-4 * np.linalg.norm(g)
    assert abs(got[0][7] - ref["nnz"]) <= max(2, 1e-6 * ref["nnz"])
