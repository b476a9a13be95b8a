"""The FP32 transfers of the mixed path over every depth of refinement, in the
middle of the box and against its far planes."""
import pytest

from tests.gpu_util import rel_l2
from tests.test_gpu_mg_levels import deep_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("level", [1, 2, 3])
def test_mixed_vcycle_over_deep_refinement(level, far):
    """The pressure of the FP64 path within the mixed path's bound (relative 1e-6), in at
    most half of Jacobi's FP32 iterations."""
    from paper_2007_02082_gb300 import IBGrid
    case = deep_case(level, far)
    kw = (dict(precision="mixed"), dict(precision="mixed", poisson_pc="jacobi"), dict(precision="fp64"))
    g = [IBGrid(case, **k) for k in kw]
    for x in g:
        x.ipcs_step(1)
    it = [x.ib_grid_info()["iters_p"] for x in g]
    assert 2 * it[0] <= it[1], it
    p = [x.ib_fields_get("P") for x in g]
    assert rel_l2(p[0], p[2]) <= 1e-6 and rel_l2(p[1], p[2]) <= 1e-6
    for x in g:
        x.close()
