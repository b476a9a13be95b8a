"""Which force systems a cluster solves and which the loop of launches (csrc/af_plan.hpp).

The expected choices are those of the faster side as measured on a GB300 where the two
differ by 15 % or more: by entries that fit the cluster's shared memories and by how far the
columns reach, not by rows alone.
"""
import os
import subprocess

import numpy as np
import pytest

from tests import force_system as F


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("plan") / "af_plan")
    subprocess.run(["g++", "-O2", "-std=c++17", "-Wall", "-I", os.path.join(F.PKG, "csrc"),
                    os.path.join(F.ROOT, "tests", "af_plan_probe.cpp"), "-o", exe], check=True)
    return exe


def route(probe, tmp_path, M, spacing, R, shuffled, cl=16):
    return route_of(probe, tmp_path, F.tube_points(M, spacing, R, shuffled=shuffled), cl)


def route_of(probe, tmp_path, X, cl=16):
    rows, rp, col, _, _, _ = F.padded([F.system(X)])
    with open(tmp_path / "sys", "wb") as f:
        np.array([rows[0], cl], np.int32).tofile(f)
        rp.tofile(f)
        col.tofile(f)
    out = subprocess.run([probe, str(tmp_path / "sys")], check=True, capture_output=True, text=True).stdout.split()
    return bool(int(out[0])), bool(int(out[1]))


@pytest.mark.parametrize("M,spacing,R,shuffled,fp32,fp64", [
    (256, 1.25, 5, False, True, True),
    (2000, 1.25, 13, False, True, True),
    (2000, 1.25, 13, True, True, None),      # FP64: 25.5 us an iteration against 24.4
    (3000, 1.25, 13, True, None, False),
    (4000, 2.4, 25, True, True, None),
    (4000, 1.25, 25, True, False, False),
    (6000, 1.25, 25, True, False, False),
    (6000, 1.25, 25, False, True, True),
    (6000, 2.4, 25, False, True, True),
    (8160, 1.25, 25, True, False, False),
    (12000, 1.25, 25, False, True, False),
    (16000, 2.4, 25, True, False, False),
    (24000, 1.25, 25, False, False, False),
    (32000, 1.25, 97, False, False, False),
    (32000, 2.4, 97, False, True, False),
    (33000, 2.4, 25, False, False, False),   # more rows than x registers
])
def test_route(probe, tmp_path, M, spacing, R, shuffled, fp32, fp64):
    got = route(probe, tmp_path, M, spacing, R, shuffled)
    assert fp32 is None or got[0] == fp32
    assert fp64 is None or got[1] == fp64


@pytest.mark.parametrize("M,spacing,R,fp32,fp64", [
    (7000, 1.8, 30, True, None),       # 11.6 us an iteration against 19.7
    (20000, 1.3, 40, False, False),    # 30.6 against 19.6
    (5000, 1.8, 25, None, True),       # 19.7 against 23.5
    (6500, 2.4, 40, None, True),       # 17.8 against 24.7
])
def test_route_of_a_sac_listed_after_its_tube(probe, tmp_path, M, spacing, R, fp32, fp64):
    """Some CTAs have no window, but few of their entries lie in others' rows."""
    got = route_of(probe, tmp_path, F.sac_points(M, spacing, R))
    assert fp32 is None or got[0] == fp32
    assert fp64 is None or got[1] == fp64


def test_no_cluster_and_smaller_clusters(probe, tmp_path):
    assert route(probe, tmp_path, 256, 2.4, 5, False, cl=0) == (False, False)
    assert route(probe, tmp_path, 4000, 2.4, 25, False, cl=8) == (True, False)   # 8 x 384 FP64 rows
