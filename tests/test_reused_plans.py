"""Plans that are reused, in every form in which their shares are held: cached with and
without pair lists, partly cached, in up to eight pieces a warp.
Every kept pair is decided by the same FP32 test on the same values however the work is
split, so at one pose the count is that of an evaluation, exactly, and both passes of an
iteration keep the same pairs."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

POSE_TOL = 1e-4


@pytest.fixture(scope="module")
def cvo():
    import __graft_entry__
    __graft_entry__.build()
    import paper_1904_02266_gb300 as m
    return m


def _wide(F, D):
    return np.ascontiguousarray(np.concatenate([F, F[:, :3] * F[:, 1:4]], 1)[:, :D])


def _near(P, seed, deg=0.2, metres=0.002):
    return synth.random_motion(np.random.default_rng(seed), deg, metres) @ P


@pytest.mark.parametrize("D", [5, 8])
def test_counts_of_reused_plans(cvo, D):
    """40k x 38k points at one lengthscale: about 100 chunks a warp, so one piece that
    overflows the cache (cost_chunk 0: few units), several pieces (48), eight (4096)."""
    d = synth.planes_pair(40000, 38011, seed=synth.seed_for(1, 41))
    FX, FZ = _wide(d["FX"], D), _wide(d["FZ"], D)
    P0, runs = _near(d["P_gt"], 5), []
    for cost_chunk in (0, 48, 4096):
        with cvo.Context(device=0, feat_dim=D, ell0=0.05, ell_min=0.05, max_iters=5, eps_pose=1e-12,
                         eps_grad=1e-12, cost_chunk=cost_chunk) as ctx:
            hx, hz = ctx.set_cloud(d["X"], FX), ctx.set_cloud(d["Z"], FZ)
            nnz = ctx.eval(hx, hz, P0, 0.05)["nnz"]
            P, st, rec = ctx.align_profile(hx, hz, P0)
            assert [r["replanned"] for r in rec] == [1, 0, 0, 0, 0]
            assert all(r["grad_pairs"] == r["step_pairs"] for r in rec)
            assert rec[0]["grad_pairs"] == nnz
            runs.append((P, [r["grad_pairs"] for r in rec]))
            # small teams: two pieces a warp, shares far beyond the cache
            with ctx.batch([hx] * 3, [hz] * 3, team_sizes=[1, 8, 33]) as b:
                Pb, sb = b.run(np.tile(P0, (3, 1, 1)))
            for p, s in zip(Pb, sb):
                assert abs(s["pair_evals"] - st["pair_evals"]) <= 3e-6 * st["pair_evals"]
                assert max(oracle.pose_error(p, P)) <= 1e-5
    for P, pairs in runs[1:]:   # poses agree to rounding, which moves a pair in a million across the cutoff
        assert max(oracle.pose_error(P, runs[0][0])) <= 1e-5
        for a, b in zip(pairs, runs[0][1]):
            assert abs(a - b) <= max(3, 3e-6 * b)


@pytest.mark.parametrize("ell_min", [0.02, 0.06])   # cached with lists, partly cached
def test_whole_solves_of_eight_features(cvo, ell_min):
    d = synth.planes_pair(12000, 11003, seed=synth.seed_for(1, 43))
    FX, FZ = _wide(d["FX"], 8), _wide(d["FZ"], 8)
    kw = dict(ell0=0.1, ell_min=ell_min, max_iters=40)
    P0 = _near(d["P_gt"], 7, 2.0, 0.02)
    with cvo.Context(device=0, feat_dim=8, **kw) as ctx:
        P, st = ctx.align(ctx.set_cloud(d["X"], FX), ctx.set_cloud(d["Z"], FZ), P0)
    ref = oracle.align(d["X"], FX, d["Z"], FZ, P0, oracle.Params(**kw))
    assert max(oracle.pose_error(P, ref["P"])) <= POSE_TOL
    assert abs(st["iters"] - ref["iters"]) <= 3
