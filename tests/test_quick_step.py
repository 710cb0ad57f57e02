"""The step tail of the solve kernel, alone (tests/quick_step.cu), against the step in FP64:
small plain steps give the passes their next pose in FP32 first (the quick step) and the
FP64 pose behind the next barrier; all others take the FP64 tail at once.

Bounds. FP64 pose: the root by Newton to 2^-40 and a rotation matrix product, 1e-11 of the
step and 1e-15 of the pose. Passes' pose: half an ulp of the rounding, as a rounded FP64 pose
has, and the change's own error: the FP32 root is off by at most its residual (4.8e-7 of
the terms, which are at most G'' / 256) and their rounding (2^-22), 3e-9 in all, and the
change is formed to about 4 x 2^-23 of itself; both times the lever, the offset of the
clouds (a quick step as wrong as 1e-7 would show)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CASE = np.dtype([("P", "f8", 16), ("cX", "f8", 3), ("cZ", "f8", 3), ("grad", "f8", 9), ("s", "f8", 7),
                 ("ell", "f8"), ("eps_pose", "f8"), ("at_floor", "i8")])
RESULT = np.dtype([("P", "f8", 16), ("tau", "f8"), ("quick", "f8"), ("R", "f4", 9), ("T", "f4", 3)])


@pytest.fixture(scope="module")
def run_steps(tmp_path_factory):
    from paper_1904_02266_gb300 import build
    lib = tmp_path_factory.mktemp("quick_step") / "quick_step.so"
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-o", str(lib), os.path.join(HERE, "quick_step.cu")], check=True)
    f = ctypes.CDLL(str(lib)).run_steps

    def run(cases):
        out = np.zeros(len(cases), RESULT)
        rc = f(cases.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p), len(cases))
        assert rc == 0
        return out
    return run


def _cases(tau, seed, offset, at_floor=0, eps_pose=1e-5):
    """Random poses, directions and quartics whose first maximiser is about tau."""
    rng = np.random.default_rng(seed)
    c = np.zeros(len(tau), CASE)
    for i, t in enumerate(tau):
        c["P"][i] = synth.random_motion(rng, rng.uniform(0, 170), rng.uniform(0, offset)).ravel()
        c["cX"][i], c["cZ"][i] = rng.uniform(-offset, offset, (2, 3))
        c["grad"][i, 0] = 100.0
        c["grad"][i, 1:7] = rng.normal(size=6) * 10.0 ** rng.uniform(-2, 3)
        s2 = -(10.0 ** rng.uniform(0, 6))
        s3, s4 = rng.normal(size=2) * abs(s2) * np.array([0.1, 0.1]) / max(t, 0.01)
        s1 = -(2 * s2 * t + 3 * s3 * t ** 2 + 4 * s4 * t ** 3)
        c["s"][i, :5] = [abs(s2), s1, s2, s3, s4]
    c["ell"], c["eps_pose"], c["at_floor"] = 0.05, eps_pose, at_floor
    return c


def _hat(w):
    return np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])


def _reference(c):
    """The step in FP64: direction, root, pose."""
    om, v = c["grad"][1:4] + np.cross(c["cX"], c["grad"][4:7]), c["grad"][4:7]
    u = np.concatenate([om, v]) / np.linalg.norm(np.concatenate([om, v]))
    k = np.array([4 * c["s"][4], 3 * c["s"][3], 2 * c["s"][2], c["s"][1]])
    r = np.roots(k)
    r = r[(abs(r.imag) < 1e-9 * abs(r.real)) & (r.real > 0)].real
    r = r[np.polyval(np.polyder(k), r) < 0]
    tau = r.min()
    for _ in range(4):
        tau -= np.polyval(k, tau) / np.polyval(np.polyder(k), tau)
    W, th = _hat(tau * u[:3]), tau * np.linalg.norm(u[:3])
    A = 1 - th ** 2 / 6 * (1 - th ** 2 / 20 * (1 - th ** 2 / 42))
    B = 0.5 * (1 - th ** 2 / 12 * (1 - th ** 2 / 30 * (1 - th ** 2 / 56)))
    C = (1 - th ** 2 / 20 * (1 - th ** 2 / 42 * (1 - th ** 2 / 72))) / 6
    E = np.eye(4)
    E[:3, :3] = np.eye(3) + A * W + B * W @ W
    E[:3, 3] = (np.eye(3) + B * W + C * W @ W) @ (tau * u[3:])
    P = E @ c["P"].reshape(4, 4)
    return tau, P, u


@pytest.mark.parametrize("offset", [0.1, 1.0, 20.0])
def test_quick_steps_are_the_fp64_step_rounded(run_steps, offset):
    tau = 10.0 ** np.linspace(-6, np.log10(1.6e-3), 400)
    cases = _cases(tau, 3, offset)
    out = run_steps(cases)
    assert (out["quick"] == 1).mean() > 0.95
    for c, r in zip(cases, out):
        t, P, u = _reference(c)
        assert abs(r["tau"] - t) <= 1e-11 * t
        lever = 1.0 + np.abs(c["cX"]).max() + np.abs(c["cZ"]).max() + np.abs(P[:3, 3]).max()
        assert np.abs(r["P"].reshape(4, 4) - P).max() <= (1e-11 * t + 2e-15) * lever
        Tc = P[:3, :3] @ c["cZ"] + P[:3, 3] - c["cX"]
        own = (3e-9 + 5e-7 * t) * (r["quick"] == 1)
        for got, want, lev in ((r["R"].reshape(3, 3), P[:3, :3], 1.0), (r["T"], Tc, 2 * lever)):
            half = 0.5 * np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
            assert (np.abs(got.astype(np.float64) - want) <= half * 1.0001 + own * lev + 1e-14 * lever).all()


def test_larger_and_stopping_steps_take_the_fp64_tail(run_steps):
    for cases in (_cases(10.0 ** np.linspace(-2.3, -0.7, 200), 5, 1.0),
                  _cases(np.full(50, 1e-5) * (1 + np.linspace(-9e-5, 9e-5, 50)), 6, 1.0, 1, 1e-5),
                  _cases(np.full(50, 3e-6), 7, 1.0, 1, 1e-5)):
        out = run_steps(cases)
        assert (out["quick"] == 0).all()
        for c, r in zip(cases, out):
            t, P, _ = _reference(c)
            assert abs(r["tau"] - t) <= 1e-10 * t
            assert np.abs(r["P"].reshape(4, 4) - P).max() <= (1e-9 * t + 1e-14) * 10
            Tc = P[:3, :3] @ c["cZ"] + P[:3, 3] - c["cX"]
            half = 0.5 * np.spacing(np.abs(Tc).astype(np.float32)).astype(np.float64)
            assert (np.abs(r["T"] - Tc) <= half * 1.0001 + 1e-8 * t + 1e-13).all()
