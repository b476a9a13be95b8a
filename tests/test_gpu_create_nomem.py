"""ib_grid_create without host memory: a status, never a C++ exception through the C entry."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import ctypes as C, sys
sys.path.insert(0, {root!r})
import workloads as W
import paper_2007_02082_gb300 as P
shim = C.CDLL({so!r})
case = W.cylinder_case(n=(8, 8, 16), length=2.0, M=60, seed=7, nu=0.1, dt=0.01)
d = P.IBGrid(case, precision="fp64")._desc
h = C.c_void_p()
shim.new_fails(1)
s = P.load_library().ib_grid_create(C.byref(d), C.byref(h))
shim.new_fails(0)
print("status", s)
"""


@pytest.mark.gpu
def test_create_does_not_throw(tmp_path):
    so = str(tmp_path / "new_fails.so")
    subprocess.run(["g++", "-O2", "-shared", "-fPIC", os.path.join(ROOT, "tests", "new_fails.cpp"), "-o", so],
                   check=True)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=ROOT, so=so)], capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert "status 0" in r.stdout
