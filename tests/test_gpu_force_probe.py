"""The cluster force solve against the loop of launches, on the same systems.

No entry point of the library lets a caller choose between the two, so a
small driver (tests/force_probe.cu) calls the library's routines.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import workloads as W
from tests import force_system as F

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    return F.build_probe(tmp_path_factory.mktemp("probe"))


# r, 1/diag and diagonal of rows 0 and 256 (two rows of different sums) for which the FP64 quotient r.z / p.q lies
# within 3e-14 of the middle between two FP32 numbers, but not so near that FP64 rounds it to the middle
EDGES = [
    ("0x1.8ef016p+0", "0x1.a69264p+0", "0x1.34e8a4p+0", "0x1.28addcp+0", "0x1.ade682p+0", "0x1.fa338cp+0"),
    ("0x1.f9aadep+0", "0x1.2037fep+0", "0x1.6246a0p+0", "0x1.e45e8ap+0", "0x1.1d4c32p+0", "0x1.8d43b2p+0"),
    ("0x1.b2ff4cp+0", "0x1.8bbc10p+0", "0x1.3cdf68p+0", "0x1.a2ed94p+0", "0x1.0c9982p+0", "0x1.b65faap+0"),
    ("0x1.f1da4ap+0", "0x1.0550e4p+0", "0x1.ec4a5ap+0", "0x1.18baa8p+0", "0x1.bada0cp+0", "0x1.290c12p+0"),
]


@pytest.mark.parametrize("cluster", [0, 8, 16])
def test_scalars_are_fp64_quotients_rounded_once(probe, tmp_path, cluster):
    """One iteration of two-row systems: x = alpha p, alpha the FP64 quotient of
    the FP64 sums rounded to FP32, each product rounded once."""
    f = np.float32
    systems, bs, dinvs, want = [], [], [], []
    for e in EDGES:
        r, d, s = ([f(float.fromhex(h)) for h in e[k:k + 2]] for k in (0, 2, 4))
        z = [r[i] * d[i] for i in (0, 1)]
        rz = sum(np.float64(r[i] * z[i]) for i in (0, 1))
        pq = sum(np.float64(z[i] * (s[i] * z[i])) for i in (0, 1))
        S = sp.csr_matrix((np.array(s, np.float64), ([0, 256], [0, 256])), shape=(257, 257))
        b, dv = np.zeros((257, 3)), np.zeros(257)
        b[[0, 256]] = np.array(r, np.float64)[:, None]
        dv[[0, 256]] = d
        systems.append(S)
        bs.append(b)
        dinvs.append(dv)
        want.append([f(rz / pq) * v for v in z])
    head, G, _ = F.solve(probe, tmp_path, systems, bs, 1, cluster, max_iter=1, dinvs=dinvs)
    for i, g in enumerate(G):
        assert list(head[i, :3]) == [1, 1, 1]
        assert np.array_equal(g[[0, 256]], np.repeat(np.array(want[i], np.float64)[:, None], 3, 1)), i


@pytest.mark.parametrize("cluster", [8, 16])
@pytest.mark.parametrize("M,spacing,shuffled", [(256, 2.4, False), (1024, 1.6, False), (1025, 1.6, False),
                                                (4096, 2.4, False), (4097, 2.4, True), (12000, 1.25, False)])
@pytest.mark.parametrize("mixed", [1, 0])
def test_cluster_and_loop_agree(probe, tmp_path, M, spacing, shuffled, cluster, mixed):
    """The same solve by a cluster and by the loop.  FP32 up to 1024 rows: every
    operation and its order are the same, so are the bits.  Else both end with a
    residual of rtol |b|: with the diagonal raised by a tenth of the largest row
    sum the condition number is below 11, so they differ by at most 2 x 11 rtol,
    and in FP32 by the rounding of some 40 iterations besides (40 x 2^-24 x 11 =
    3e-5 each)."""
    if not mixed and M > 384 * cluster:
        pytest.skip("FP64 clusters take at most 384 rows a CTA")
    S = F.system(F.tube_points(M, spacing, 13 if M < 4000 else 25, shuffled=shuffled), shift=0.1)
    b = np.random.default_rng(M).normal(size=(M, 3))
    kw = dict(rtol=1e-12 if not mixed else 0.0, rtol_inner=1e-5)
    ha, (a,), _ = F.solve(probe, tmp_path, [S], [b], mixed, cluster, **kw)
    hl, (l,), _ = F.solve(probe, tmp_path, [S], [b], mixed, 0, **kw)
    assert ha[0, :3].min() > 3 and np.abs(ha[0, :3] - hl[0, :3]).max() <= 1
    if mixed and M <= 1024:
        assert np.array_equal(a, l)
    tol = 22e-5 + 6e-5 if mixed else 22e-12
    assert np.all(np.linalg.norm(a - l, axis=0) <= tol * np.linalg.norm(l, axis=0))


@pytest.mark.parametrize("mixed", [1, 0])
def test_library_routes_problems_of_a_batch_apart(probe, tmp_path, mixed):
    """A problem of the loop's (points in random order) between two of the clusters':
    the library's choice gives each the bits it has alone."""
    systems = [F.system(F.tube_points(M, 1.6, R, shuffled=s), shift=0.1)
               for M, R, s in ((700, 13, False), (8160, 25, True), (2000, 13, False))]
    bs = [np.random.default_rng(S.shape[0]).normal(size=(S.shape[0], 3)) for S in systems]
    kw = dict(rtol=1e-12 if not mixed else 0.0, rtol_inner=1e-5)
    head, G, _ = F.solve(probe, tmp_path, systems, bs, mixed, -1, **kw)
    for i, (S, b) in enumerate(zip(systems, bs)):
        ha, (a,), _ = F.solve(probe, tmp_path, [S], [b], mixed, 0 if i == 1 else 16, **kw)
        assert np.array_equal(head[i, :3], ha[0, :3]) and np.array_equal(G[i], a), i


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_batch_with_a_loop_member(precision):
    """Steps of a batch whose second member's force system goes to the loop (8160
    points in random order) and the others' to clusters: each member as alone."""
    from paper_2007_02082_gb300 import IBBatch, IBGrid
    mid = W.cylinder_case(n=(32, 32, 128), M=8160, seed=92, nu=0.05, dt=0.005)
    k = np.random.default_rng(5).permutation(len(mid["X"]))
    mid["X"], mid["dS"], mid["UB"] = (np.ascontiguousarray(mid[f][k]) for f in ("X", "dS", "UB"))
    cases = [W.cylinder_case(n=(8, 8, 16), length=2.0, M=270, seed=91, nu=0.1, dt=0.01), mid,
             W.cylinder_refined_small(n=(16, 16, 20), seed=93)]
    alone = []
    for c in cases:
        g = IBGrid(c, precision=precision)
        g.ipcs_step(2)
        alone.append([g.ib_fields_get(f) for f in ("U", "P", "F_LAG")])
        g.close()
    mem = [IBGrid(c, precision=precision, deferred=True) for c in cases]
    b = IBBatch(mem)
    assert np.all(b.step(2) == 0)
    for i, m in enumerate(mem):
        for f, ref in zip(("U", "P", "F_LAG"), alone[i]):
            assert np.array_equal(m.ib_fields_get(f), ref), (i, f)
    b.close()
    for m in mem:
        m.close()
