"""Grid reductions around their group edges (32 CTAs a group, 32 groups a warp pass).

A member with more than 32 chunks next to members with fewer, none of whose
CTA counts is a multiple of 32, so that groups start at every offset: every
member keeps its bits alone, in the mix and under the other chunk size.
"""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_groups_follow_the_instance(precision):
    from paper_2007_02082_gb300 import IBBatch, IBGrid
    cases = [W.cylinder_case(n=(9, 9, 15), length=2.0, M=120, seed=41, nu=0.05, dt=0.01),
             W.cylinder_case(n=(42, 44, 90), length=4.0, M=900, seed=42, nu=0.05, dt=0.01),      # 432 bricks
             W.cylinder_refined_small(n=(16, 16, 20), seed=43),
             W.cylinder_case(n=(8, 8, 16), length=2.0, M=120, seed=44, nu=0.05, dt=0.01)]
    for tune in ({}, {"stream_chunk": 4}):
        alone = []
        for c in cases:
            g = IBGrid(c, precision=precision, tune=tune)
            g.ipcs_step(2)
            alone.append((g.ib_fields_get("U"), g.ib_fields_get("P")))
            g.close()
        mem = [IBGrid(c, precision=precision, deferred=True, tune=tune) for c in cases]
        assert mem[1].ib_grid_info()["n_bricks"] > 33 * 8
        b = IBBatch(mem)
        assert np.all(b.step(2) == 0)
        for i, m in enumerate(mem):
            assert np.array_equal(m.ib_fields_get("U"), alone[i][0]), i
            assert np.array_equal(m.ib_fields_get("P"), alone[i][1]), i
        b.close()
        for m in mem:
            m.close()
