"""The weight of active source groups in the rebalanced work split (csrc/split_rule.h,
compiled for the host): it must hang on what fits a warp's cache, so on the feature width,
and not on the units in which the caller's cost model counts work. The rows are shares that
the kernel's first split of room pairs measured on 152 blocks (cost_chunk 48, cost_cluster
32): features, cache floats a warp, points, clusters, units a warp, warps, weight."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
ROWS = [(5, 2592, 10000, 3258, 131, 2280, 12), (5, 2592, 15000, 3729, 180, 2280, 24),
        (5, 2592, 20000, 4038, 232, 2280, 24), (5, 2592, 28000, 4316, 315, 2280, 24),
        (5, 2592, 34000, 5989, 797, 2432, 12), (8, 2592, 15000, 3729, 180, 2280, 24),
        (8, 2592, 20000, 4038, 232, 2280, 24), (8, 2592, 28000, 4316, 315, 2280, 12),
        (8, 2592, 34000, 5989, 798, 2432, 12), (3, 2752, 28000, 4316, 315, 2280, 24),
        (3, 2752, 34000, 5989, 797, 2432, 12), (0, 2848, 28000, 4316, 315, 2280, 24),
        (0, 2848, 45000, 6415, 1223, 2432, 12)]


@pytest.fixture(scope="module")
def weight(tmp_path_factory):
    d = tmp_path_factory.mktemp("split_rule")
    src, lib = d / "rule.cpp", d / "rule.so"
    src.write_text('#include "paper_1904_02266_gb300/csrc/split_rule.h"\n'
                   'extern "C" int weight(long long total, long long warps, int ncl, int points,\n'
                   '                      int chunk, int cluster, int floats, int cap) {\n'
                   '  return cvo::active_weight(total, warps, ncl, points, chunk, cluster, floats, cap);\n}\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", ROOT, str(src), "-o", str(lib)],
                   check=True)
    f = ctypes.CDLL(str(lib)).weight
    f.argtypes = [ctypes.c_longlong] * 2 + [ctypes.c_int] * 6
    return f


@pytest.mark.parametrize("D,cap,points,ncl,share,warps,want", ROWS)
def test_measured_shares(weight, D, cap, points, ncl, share, warps, want):
    assert weight(share * warps, warps, ncl, points, 48, 32, 4 + D, cap) == want


@pytest.mark.parametrize("D,cap,points,ncl,share,warps,want", ROWS)
def test_the_unit_of_work_does_not_matter(weight, D, cap, points, ncl, share, warps, want):
    """The same chunks and clusters under other costs."""
    size = points / ncl + 1.5
    chunks = (share * warps - 32 * ncl) / (size + 48)
    for cost_chunk in (0, 16, 96, 256, 4096):
        for cost_cluster in (0, 128, 65536):
            total = round(chunks * (size + cost_chunk) + ncl * cost_cluster)
            assert weight(total, warps, ncl, points, cost_chunk, cost_cluster, 4 + D, cap) == want


def test_wider_features_never_get_the_heavier_weight_alone(weight):
    """The largest mean share that is weighed heavily takes the same part of the cache."""
    for points, ncl in ((20000, 4000), (8000, 900), (60000, 2500)):
        top = {}
        for D, cap in ((0, 2592), (3, 2592), (5, 2592), (8, 2592)):
            heavy = [s for s in range(60, 4000) if weight(s * 2280, 2280, ncl, points, 48, 32, 4 + D, cap) == 24]
            top[D] = (heavy[-1] - 32 * ncl / 2280) / (points / ncl + 49.5) * 32 * (4 + D) + \
                (points / ncl + 1.5) * ncl / 2280 * (4 + D)
        for D in top:
            assert abs(top[D] - 0.7 * 2592) < 2 * 32 * (4 + D) / 30, (points, top)
