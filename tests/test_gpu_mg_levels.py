"""Transfers between the composite grid and G0 over every depth of refinement.

The restriction halves a brick once per level (8 -> 5 -> 3 -> 2 nodes an axis), the
prolongation takes its weights once per level except in bricks at the far planes;
a transfer that is not the other's transpose, or not the interpolation of the
nested meshes, costs the V-cycle its hold on the iteration count or the solve its
convergence.
"""
import numpy as np
import pytest

import workloads as W
from tests.gpu_util import rel_l2

pytestmark = pytest.mark.gpu


def deep_case(level, far=False):
    """A small sphere of points in the middle (or against the far planes) of a
    box of 8 x 8 x 16 cells: bricks on every level from 0 to level."""
    n, ext = (8, 8, 16), (1.0, 1.0, 2.0)
    h = 1.0 / (8 << level)
    k = np.arange(60)
    z = 1.0 - (2.0 * k + 1.0) / 60.0
    a = np.pi * (1.0 + 5.0 ** 0.5) * k
    s = np.sqrt(1.0 - z * z)
    c = np.array([1.0 - 6 * h, 0.5, 2.0 - 6 * h]) if far else np.array([0.49, 0.52, 1.03])
    X = c + 2.0 * h * np.stack([s * np.cos(a), s * np.sin(a), z], axis=1)
    return {"origin": (0.0, 0.0, 0.0), "extent": ext, "n": n, "max_level": level, "refine_band": 1,
            "reduce_band": -1, "nu": 0.1, "rho": 1.0, "dt": 0.01,
            "ports": [W._port(2, 0, (0.5, 0.5, 0.0), 0.499, W.PINLET, a0=1.0),
                      W._port(2, 1, (0.5, 0.5, 2.0), 0.499, W.OUTLET)],
            "X": X, "dS": np.full(60, 4.0 * np.pi * (2.0 * h) ** 2 / 60), "UB": np.zeros((60, 3)),
            "inside": np.ones((n[2], n[1], n[0]), np.uint8)}


@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("level", [1, 2, 3])
def test_vcycle_over_deep_refinement(level, far):
    """Same pressure as with Jacobi to the solve tolerance (1e-10 relative
    residual against a condition number below 1e2 of the preconditioned
    operator: 1e-8), in at most half of the iterations."""
    from paper_2007_02082_gb300 import IBGrid
    case = deep_case(level, far)
    a = IBGrid(case, precision="fp64")
    b = IBGrid(case, precision="fp64", poisson_pc="jacobi")
    a.ipcs_step(1)
    b.ipcs_step(1)
    ia, ib_ = a.ib_grid_info(), b.ib_grid_info()
    assert 2 * ia["iters_p"] <= ib_["iters_p"], (ia["iters_p"], ib_["iters_p"])
    assert rel_l2(a.ib_fields_get("P"), b.ib_fields_get("P")) < 1e-8
    a.close()
    b.close()
