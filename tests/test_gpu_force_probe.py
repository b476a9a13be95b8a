"""The cluster force solve against the loop of launches, on the same systems.

No entry point of the library lets a caller choose between the two, so a
small driver (tests/force_probe.cu) calls the library's routines.
"""
import numpy as np
import pytest
import scipy.sparse as sp

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
