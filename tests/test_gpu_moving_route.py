"""A moving wall whose points change the force solver: ordered along the wall they
go to a cluster, in random order to the loop of launches."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("U", "P", "F_LAG")


def _case():
    case = W.cylinder_case(n=(32, 32, 64), length=2.0, M=4000, seed=94, nu=0.05, dt=0.005)
    X = np.asarray(case["X"])
    Xp = np.ascontiguousarray(X[np.random.default_rng(6).permutation(len(X))])
    assert np.ptp(case["dS"]) == 0     # the points take one another's places: the grid stays the same
    return case, X, Xp


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("moves", [1, 2])
def test_moved_points_choose_as_a_fresh_handle(precision, moves):
    """Into random order, and back: the handle steps bitwise like a fresh one."""
    from paper_2007_02082_gb300 import IBGrid
    case, X, Xp = _case()
    g = IBGrid(case, precision=precision)
    for k in range(moves):
        g.ib_set_points((Xp, X)[k])
    h = IBGrid(dict(case, X=(Xp, X)[moves - 1]), precision=precision)
    for x in (g, h):
        x.ipcs_step(2)
    for f in FIELDS:
        assert np.array_equal(g.ib_fields_get(f), h.ib_fields_get(f)), f
    g.close()
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_captured_steps_follow_the_choice(precision):
    """Order and disorder in turn between steps: the captured graphs step
    bitwise like launches issued one by one."""
    from paper_2007_02082_gb300 import IBGrid
    case, X, Xp = _case()
    g, e = IBGrid(case, precision=precision), IBGrid(case, precision=precision, profile=True)
    for pts in (X, Xp, X, X, Xp, Xp):
        for x in (g, e):
            x.ib_set_points(pts)
            x.ipcs_step(1)
        for f in FIELDS:
            assert np.array_equal(g.ib_fields_get(f), e.ib_fields_get(f)), f
    g.close()
    e.close()
