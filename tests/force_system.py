"""Force systems S G = b for tests, and the probe that solves them with the library.

S = W W^T from the four-point kernel's weights of points on a tube wall in a
uniform unit grid, every support node free.
"""
import os
import shutil
import subprocess

import numpy as np
import scipy.sparse as sp

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
PKG = os.path.join(ROOT, "paper_2007_02082_gb300")


def tube_points(M, spacing, R, seed=3, shuffled=False):
    """M points on a tube of R cells, ring by ring along its axis, or in random order."""
    rng = np.random.default_rng(seed)
    n = max(8, int(round(2 * np.pi * R / spacing)))
    rings = -(-M // n)
    s = spacing * (np.arange(rings)[:, None] + 0.5 + rng.uniform(-0.35, 0.35, (rings, n)))
    t = 2 * np.pi / n * (np.arange(n)[None] + 0.5 + rng.uniform(-0.35, 0.35, (rings, n)))
    X = np.stack([R + 4 + R * np.cos(t), R + 4 + R * np.sin(t), 4 + s], -1).reshape(-1, 3)[:M]
    return X[rng.permutation(M)] if shuffled else X


def sac_points(M, spacing, R, seed=3):
    """A tube's points, ring by ring, then those of a sphere of 1.2 R halfway along it
    that lie outside the tube: rows next to one another on the wall far apart in the list."""
    rng = np.random.default_rng(seed)
    m = 3 * M // 10
    X = tube_points(M - m, spacing, R, seed)
    k = np.arange(4 * m)
    z, a = 1 - (2 * k + 1) / (4.0 * m), np.pi * (1 + 5 ** 0.5) * k
    s = np.sqrt(1 - z * z)
    c = np.array([R + 4 + 1.4 * R, R + 4, 4 + 0.5 * (X[-1, 2] - 4)])
    N = np.stack([s * np.cos(a), s * np.sin(a), z], -1)
    Y = c + 1.2 * R * N
    Y = Y[np.hypot(Y[:, 0] - R - 4, Y[:, 1] - R - 4) > R]
    near = np.linalg.norm(X - c, axis=1) > 1.2 * R
    return np.concatenate([X[near], Y[np.sort(rng.permutation(len(Y))[:m])]])


def _phi(r):
    r = np.abs(r)
    a = (3 - 2 * r + np.sqrt(np.maximum(1 + 4 * r - 4 * r * r, 0))) / 8
    b = (5 - 2 * r - np.sqrt(np.maximum(-7 + 12 * r - 4 * r * r, 0))) / 8
    return np.where(r <= 1, a, np.where(r <= 2, b, 0.0))


def system(X, shift=0.0):
    """S as CSR with the library's pattern (supports that share a node), plus
    shift times its largest row sum on the diagonal."""
    a = np.arange(64)
    q = (np.floor(X).astype(int) - 1)[:, None] + np.stack([a & 3, a >> 2 & 3, a >> 4], -1)[None]
    w = _phi(q - X[:, None]).prod(-1)
    n = q.reshape(-1, 3).max(0) + 1
    _, col = np.unique((q[..., 2] * n[1] + q[..., 1]) * n[0] + q[..., 0], return_inverse=True)
    at = (np.repeat(np.arange(len(X)), 64), col.ravel())
    W = sp.csr_matrix((w.ravel(), at))
    one = sp.csr_matrix((np.full(w.size, 1e-150), at))
    S = (W @ W.T + one @ one.T).tocsr()
    S = (S + shift * abs(S).sum(1).max() * sp.identity(len(X))).tocsr()
    S.sort_indices()
    return S


def padded(systems, bs=None, dinvs=None):
    """Rows of the problems one after another, each padded to whole blocks of
    256: rows, rowptr, col, val, dinv, b."""
    rows = [-(-S.shape[0] // 256) * 256 for S in systems]
    rp, col, val = [np.zeros(1, np.int64)], [], []
    dinv, b = np.zeros(sum(rows)), np.zeros((sum(rows), 3))
    R0 = 0
    for i, (S, m) in enumerate(zip(systems, rows)):
        n = S.shape[0]
        rp.append(rp[-1][-1] + S.indptr[1:])
        rp.append(np.full(m - n, rp[-1][-1]))
        rp = [np.concatenate(rp)]
        col.append(S.indices + R0)
        val.append(S.data)
        dinv[R0:R0 + n] = 1.0 / S.diagonal() if dinvs is None else dinvs[i]
        if bs is not None:
            b[R0:R0 + n] = bs[i]
        R0 += m
    return rows, rp[0].astype(np.int32), np.concatenate(col).astype(np.int32), np.concatenate(val), dinv, b


def build_probe(path):
    """Compile tests/force_probe.cu against the built library."""
    nvcc = os.environ.get("NVCC") or shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    lib, exe = os.path.join(PKG, "lib"), os.path.join(str(path), "force_probe")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-cudart", "shared",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"),
                    os.path.join(ROOT, "tests", "force_probe.cu"), "-o", exe, "-L", lib, "-libgpu",
                    "-Xlinker", "-rpath," + lib], check=True)
    return exe


def solve(exe, tmp, systems, bs, mixed, cluster, max_iter=2000, max_outer=1, rtol=0.0, rtol_inner=0.0, dinvs=None,
          reps=1):
    """Solve with clusters of `cluster` CTAs (0: the loop of launches, -1: the
    library's choice): per problem (iterations, status), G, seconds."""
    rows, rp, col, val, dinv, b = padded(systems, bs, dinvs)
    src, dst = os.path.join(str(tmp), "in"), os.path.join(str(tmp), "out")
    with open(src, "wb") as f:
        np.array([len(systems), mixed, cluster, max_iter, max_outer, reps], np.int64).tofile(f)
        np.array([rtol, rtol_inner]).tofile(f)
        np.array(rows, np.int64).tofile(f)
        for a in (rp, col, val, dinv, b, np.zeros_like(b)):
            a.tofile(f)
    subprocess.run([exe, src, dst], check=True, timeout=120)
    with open(dst, "rb") as f:
        head = np.fromfile(f, np.int32, 5 * len(systems)).reshape(-1, 5)
        G = np.fromfile(f, np.float64, b.size).reshape(b.shape)
        sec = np.fromfile(f, np.float64, reps)
    R0, out = 0, []
    for S, m in zip(systems, rows):
        out.append(G[R0:R0 + S.shape[0]])
        R0 += m
    return head, out, sec
