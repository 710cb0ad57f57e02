"""The work split in pieces from all over the cloud: teams of one block to the
whole GPU cut the same pair into 16 to 9728 pieces, one to four per warp, over
single-use and reused plans, and must find the same pairs and the same pose.
Every kept pair is decided by the same FP32 test whatever the split, so the
counts of the first iteration are equal; poses agree to the parity bar of FP32
sums taken in another order (steps of at most about 0.2, sums good to about 1e-6:
1e-5 rad and m after three iterations)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cvo():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1904_02266_gb300 as m
    return m


@pytest.mark.parametrize("n,m", [(1, 1), (40, 33), (700, 900), (9000, 8001)])
@pytest.mark.parametrize("kw", [{}, {"ell0": 0.05, "ell_min": 0.05}, {"feat_dim": 8, "color_mode": 2,
                                                                     "color_scale": 1.0}])
def test_pieces_cover_the_work(cvo, n, m, kw):
    d = synth.planes_pair(n, m, seed=synth.seed_for(1, n % 89))
    rng = np.random.default_rng(3)
    D = kw.get("feat_dim", 5)
    FX, FZ = (rng.random((k, D)).astype(np.float32) for k in (n, m))
    pairs, poses = [], []
    for iters in (1, 3):
        with cvo.Context(device=0, max_iters=iters, **kw) as ctx:
            hx, hz = ctx.set_cloud(d["X"], FX), ctx.set_cloud(d["Z"], FZ)
            runs = [ctx.align(hx, hz, d["P_gt"])]
            teams = [1, 2, 3, 19, 33]
            with ctx.batch([hx] * 5, [hz] * 5, team_sizes=teams) as b:
                P, st = b.run(np.tile(d["P_gt"], (5, 1, 1)))
            runs += list(zip(P, st))
        if iters == 1:
            pairs = [s["pair_evals"] for _, s in runs]
        poses = [p for p, _ in runs]
    assert len(set(pairs)) == 1, pairs
    assert pairs[0] > 0 or n < 100
    for p in poses[1:]:
        ang, tr = oracle.pose_error(p, poses[0])
        assert ang <= 1e-5 and tr <= 1e-5, (ang, tr)
