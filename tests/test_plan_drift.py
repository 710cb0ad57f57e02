"""The drift test behind reused plans as the solve kernel forms it: differences of the FP32
poses that the plan and the passes use (tests/test_plan_superset.py takes them between
FP64 poses), the rest in FP32 with 2e-5 relative and 1e-6 r_c margins. A pose that passes keeps
every pair of the pass inside the plan radius at the plan pose, with translations of up to
several hundred cutoff radii, whose FP32 rounding moves the points by more than the pose's
own differences do, and with poses an ulp off the rounded FP64 pose, as an FP32 step leaves
them. No GPU."""
import numpy as np
import pytest

from test_plan_superset import F, fmaf, listed, pass_keeps, rot, transform


def drift_ok(R, T, Rq, Tq, need, rp, src_radius_f):
    d = np.concatenate([(R - Rq).ravel(), T - Tq])
    assert d.dtype == F
    sq = np.zeros(16, F)   # lanes 4 r + c, as the warp holds the 3 x 4 pose
    for r in range(3):
        sq[4 * r:4 * r + 3] = d[3 * r:3 * r + 3] * d[3 * r:3 * r + 3]
        sq[4 * r + 3] = d[9 + r] * d[9 + r]
    rot_lane = np.array([i < 12 and i % 4 != 3 for i in range(16)])
    sums = []
    for lanes in (rot_lane, ~rot_lane):
        v = np.where(lanes, sq, F(0))
        for off in (8, 4, 2, 1):
            v = (v + v[np.arange(16) ^ off]).astype(F)
        sums.append(v[0])
    drift = F(fmaf(np.sqrt(sums[0]), src_radius_f, np.sqrt(sums[1])) * F(1 + 2e-5))
    drift = fmaf(F(1e-6), need, drift)
    return bool(F(need + drift) <= rp), drift


def _case(seed, ell, radius, shift, drift_frac, ulps):
    rng = np.random.default_rng(seed)
    z = (rng.normal(size=(300, 3)) * radius / 2).clip(-radius, radius).astype(F)
    rc = np.sqrt(2 * ell * ell * np.log(1000.0))
    rc2 = F(rc * rc)
    need = F(np.sqrt(np.float64(rc2)) * 1.001)
    rp = F(np.float64(need) * 1.1)
    src_radius_f = F(F(np.linalg.norm(np.abs(z).max(axis=0).astype(np.float64))) * F(1 + 1e-6))
    Rp = rot(rng.normal(size=3), rng.uniform(0, np.pi))
    Tp = rng.normal(size=3)
    Tp *= shift / np.linalg.norm(Tp)
    allow = float(rp - need)
    share = rng.uniform(0.2, 0.8)
    dR = rot(rng.normal(size=3), share * drift_frac * allow / (np.sqrt(2.0) * float(src_radius_f)))
    dT = rng.normal(size=3)
    dT *= (1 - share) * drift_frac * allow / np.linalg.norm(dT)
    Rc, Tc = dR @ Rp, Tp + dT
    poses = [v.astype(F) for v in (Rp, Tp, Rc, Tc)]
    if ulps:   # as far off the rounded pose as an FP32 step leaves it
        poses = [np.nextafter(v, rng.choice([-F(9), F(9)], v.shape) * 1000).astype(F) for v in poses]
    Rpf, Tpf, Rcf, Tcf = poses
    ok, _ = drift_ok(Rcf, Tcf, Rpf, Tpf, need, rp, src_radius_f)
    kept = missed = 0
    for j in range(len(z)):
        zt, zp = transform(Rcf, Tcf, z[j]), transform(Rpf, Tpf, z[j])
        o = (zt + rng.uniform(-rc, rc, size=3)).astype(F)
        for _ in range(8):
            u = rng.normal(size=3)
            x = (zt + u / np.linalg.norm(u) * rc * rng.uniform(0.97, 1.0)).astype(F)
            if pass_keeps(x, zt, o, rc2):
                kept += 1
                missed += 0 if listed(x, zp, F(rp * rp)) else 1
    return ok, kept, missed


@pytest.mark.parametrize("ulps", [0, 1])
@pytest.mark.parametrize("ell,radius,shift", [(0.02, 5.0, 0.1), (0.02, 5.0, 25.0), (0.02, 25.0, 25.0),
                                              (0.05, 5.0, 60.0), (0.15, 3.0, 200.0)])
def test_a_pose_that_passes_keeps_its_pairs(ell, radius, shift, ulps):
    ok, kept, missed = _case(11, ell, radius, shift, 0.95, ulps)
    assert ok
    assert kept > 1000
    assert missed == 0, (missed, kept)


@pytest.mark.parametrize("shift", [0.1, 25.0])
def test_drift_beyond_the_skin_is_refused_and_would_miss_pairs(shift):
    ok, kept, missed = _case(5, 0.02, 5.0, shift, 3.0, 0)
    assert not ok
    assert missed > 0, kept


def test_an_unchanged_pose_has_no_drift():
    R, T = rot(np.array([1.0, 2.0, 3.0]), 0.7).astype(F), np.array([25.0, -3.0, 8.0], F)
    ok, drift = drift_ok(R, T, R, T, F(0.07441), F(0.08185), F(5.0))
    assert ok and drift <= F(1.01e-6) * F(0.07441)
