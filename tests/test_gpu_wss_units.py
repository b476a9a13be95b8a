"""Wall shear stress in any unit of length (ib_wss, Sec. 2.6)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [-73, -40, 40, 62])
def test_wss_scales_with_the_unit_of_length(k):
    """All lengths times 2^k, the velocities as they are: every rounding of FP64 is
    the same up to that power of two, so the velocity gradient is 2^-k times
    that of k = 0 to the last bit.  At 2^-73 the squared distances lie among the
    denormal FP32 numbers, at 2^62 near the largest."""
    from paper_2007_02082_gb300 import IBGrid
    got = []
    for s in (1.0, 2.0 ** k):
        c = W.cylinder_case(n=(12, 14, 9), length=1.5, M=70, seed=80, nu=0.05, dt=0.01)
        for f in ("origin", "extent"):
            c[f] = tuple(v * s for v in c[f])
        c["X"], c["dS"] = c["X"] * s, c["dS"] * s * s
        c["ports"] = [dict(p, center=tuple(v * s for v in p["center"]), radius=p["radius"] * s) for p in c["ports"]]
        g = IBGrid(c, precision="fp64")
        u = np.random.default_rng(3).standard_normal((g.ib_grid_info()["n_nodes"], 3))
        g.ib_fields_set("U", u)
        n = np.array(c["X"])
        n[:, 2] = 0
        n /= np.hypot(n[:, 0], n[:, 1])[:, None]
        got.append(g.ib_wss(n, with_grad=True)[1] * s)
        g.close()
    assert np.array_equal(got[0], got[1])
