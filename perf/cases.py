"""What a user of the library has it do, as cases that can be timed and compared.

A pass is one time step of a handle or of a batch with its velocity and
pressure read back to the device (the loop of every simulation), the same with
the wall moved first, or one evaluation of the wall shear stress.  Vessels are
seeded synthetic ones (a straight tube, a 90-degree bend, a tube with a sac)
started from rest with a pulsating inflow, as the repository's tests, benchmark
and serving mix make them: uniform and refined grids, odd cell counts, velocity
and pressure inlets, both viscous forms, both precisions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2007_02082_gb300 import IBBatch, IBGrid

# Keys of a case:
#   call        "step", "move" (new wall points, then a step), "wss", "batch"
#   kind        "tube" (R 0.5 in a box 1.2 wide), "bend", "sac"; a batch cycles through all three
#   n           coarse cells per 1.2 units of length (the tube's box width); z_cells along the tube
#   length      length of the tube (legs of the bend, tube of the sac)
#   levels      refinement levels in the wall band (0: uniform, whole box for the tube)
#   spacing     distance of the wall points in finest cells
#   nu, cfl     viscosity; dt = cfl x the finest spacing
#   inlet, viscous, precision; members and cells_lo of a batch
_BASE = dict(call="step", kind="tube", n=16, z_cells=64, length=4.0, levels=0, spacing=1.27, nu=0.1, cfl=0.16,
             inlet="velocity", viscous="grad", precision="mixed", members=1)


def _with(name=None, **kw):
    c = dict(_BASE, **kw)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest problem anybody steps (a quick look at a set-up): launches and latency are all there is
        _with("tube_8x8x16_mixed", n=8, z_cells=16, length=2.0, spacing=1.25),
        # the Poiseuille tube of the validation runs, plain FP64, wall points at the spacing rule of the method
        _with("tube_16x16x64_fp64", precision="fp64"),
        # the same tube refined twice over: dense wall points make the force system the longest solve
        _with("tube_32x32x128_dense_mixed", n=32, z_cells=128, nu=0.05, spacing=1.25),
        # the refined tube, the ordinary production size, in both precisions
        _with("tube_64x64x256_L1_mixed", n=64, z_cells=256, levels=1, spacing=2.53, nu=0.02, cfl=0.256),
        _with("tube_64x64x256_L1_fp64", n=64, z_cells=256, levels=1, spacing=2.53, nu=0.02, cfl=0.256,
              precision="fp64"),
        # pressure-driven, symmetric viscous form, cell counts that fit no tile
        _with("tube_33x33x131_L1_pressure_sym", n=33, z_cells=131, levels=1, spacing=2.4, nu=0.03, cfl=0.2,
              inlet="pressure", viscous="sym"),
        # a pulsating wall: the points move before every step
        _with("tube_41x41x150_L1_moving", call="move", n=41, z_cells=150, levels=1, spacing=2.4, nu=0.03, cfl=0.2),
        # serving: eight small requests of different shapes and depths in one batch
        _with("batch_8_requests", call="batch", kind="mix", n=20, z_cells=60, length=3.0, spacing=2.3, nu=0.04,
              cfl=0.25, members=8, levels=2),
        # post-processing of a run: wall shear stress at every wall point
        _with("wss_tube_64x64x256_L1", call="wss", n=64, z_cells=256, levels=1, spacing=2.53, nu=0.02, cfl=0.256,
              precision="fp64"),
        # the large one: two levels, 15 million leaf cells
        _with("sac_L2_15M_mixed", kind="sac", n=58, length=4.0, levels=2, spacing=4.3, nu=0.01, cfl=0.192),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choices(["step", "move", "wss", "batch"], [7, 1, 1, 1])[0]
    c = dict(_BASE, call=call)
    c["kind"] = "tube" if call in ("move", "wss") else "mix" if call == "batch" else rng.choice(["tube", "bend", "sac"])
    c["levels"] = rng.choice([1, 1, 2]) if call != "step" else rng.choice([0, 1, 1, 2])
    c["length"] = round(rng.uniform(2.0, 4.0), 3)
    c["precision"] = "fp64" if call == "wss" or (call == "step" and rng.random() < 0.25) else "mixed"
    hi = {0: 60, 1: 64, 2: 32}[c["levels"]] if c["precision"] == "mixed" else {0: 44, 1: 44, 2: 20}[c["levels"]]
    if call == "batch":
        c["members"] = rng.randint(2, 8)
        hi = 22
    c["n"] = log_int(8 if c["levels"] == 0 else 14, hi)
    c["z_cells"] = max(8, int(round(c["n"] * c["length"] / 1.2 * rng.uniform(0.9, 1.25))))
    c["spacing"] = round(rng.uniform(1.25, 2.4) if c["levels"] == 0 else rng.uniform(2.2, 2.6), 3)
    # cell Reynolds number of the coarse cells below 2: the convection is not stabilised
    c["nu"] = round(min(0.1, max(0.01, 1.2 / c["n"] * rng.uniform(0.6, 1.3))), 5)
    c["cfl"] = round(rng.uniform(0.13, 0.25), 4)
    if call == "step" and c["kind"] == "tube" and rng.random() < 0.4:
        c["inlet"] = "pressure"
        c["viscous"] = rng.choice(["grad", "sym"])
    return c


# ---------------------------------------------------------------------------
# Geometry: the dictionaries that IBGrid takes
# ---------------------------------------------------------------------------
def _strata(rng, n_s, n_t):
    """One point per cell of an n_s x n_t grid of the unit square, off its centre by at most 0.35 of a cell."""
    s = (np.arange(n_s)[:, None] + 0.5 + rng.uniform(-0.35, 0.35, (n_s, n_t))) / n_s
    t = (np.arange(n_t)[None, :] + 0.5 + rng.uniform(-0.35, 0.35, (n_s, n_t))) / n_t
    return s.ravel(), t.ravel()


def _vessel(case, rng):
    """The problem of one case: box, wall points with normals, inside mask, ports, parameters."""
    kind, L, R = case["kind"], float(case["length"]), 0.5
    h = 1.2 / case["n"]
    scale = 1 << case["levels"]
    if kind == "tube":
        lo, n = (-0.6, -0.6, 0.0), (case["n"], case["n"], case["z_cells"])
        ext = (1.2, 1.2, L)
    elif kind == "bend":   # up along z, a quarter torus of centreline radius 1.25, out along x
        leg, rc = 0.3 * L, 1.25
        lo, n = (-R - 4 * h, -R - 4 * h, 0.0), None
        hi = (rc + leg, R + 4 * h, leg + rc + R + 4 * h)
    else:                  # a tube with a sphere of radius 0.6 centred 0.7 off its axis
        rs, off = 0.6, 0.7
        lo, n = (-R - 4 * h, -rs - 4 * h, 0.0), None
        hi = (off + rs + 4 * h, rs + 4 * h, L)
    if n is None:
        n = tuple(max(4, int(math.ceil((hi[a] - lo[a]) / h - 1e-9))) for a in range(3))
        ext = [n[a] * h for a in range(3)]
        out = 0 if kind == "bend" else 2
        ext[out] = hi[out] - lo[out]      # the outlet lies on this face
        ext = tuple(ext)
    hc = [ext[a] / n[a] for a in range(3)]
    hf = min(hc) / scale
    d = case["spacing"] * hf
    lay = np.random.default_rng(7)      # the layout of the points belongs to the case, not to the seed
    th_n = max(8, int(round(2 * math.pi * R / d)))
    z, y, x = np.meshgrid(*[lo[a] + (np.arange(n[a]) + 0.5) * hc[a] for a in (2, 1, 0)], indexing="ij")

    def tube(length):
        s, t = _strata(lay, max(4, int(round(length / d))), th_n)
        th = 2 * math.pi * t
        N = np.stack([np.cos(th), np.sin(th), 0 * th], 1)
        return np.stack([R * N[:, 0], R * N[:, 1], length * s], 1), N, np.full(len(s), 2 * math.pi * R * length / len(s))

    if kind == "tube":
        X, N, dS = tube(L)
        inside = np.hypot(x, y) < R
        outlet = (2, 1, (0.0, 0.0, L))
    elif kind == "sac":
        X, N, dS = tube(L)
        c0 = np.array([off, 0.0, 0.5 * L])
        keep = np.linalg.norm(X - c0, axis=1) > rs
        m_n = max(4, int(round(math.sqrt(2 * math.pi) * rs / d)))
        s, t = _strata(lay, m_n, 2 * m_n)
        mu, ph = 2 * s - 1, 2 * math.pi * t
        Ns = np.stack([np.sqrt(1 - mu * mu) * np.cos(ph), np.sqrt(1 - mu * mu) * np.sin(ph), mu], 1)
        Xs = c0 + rs * Ns
        ks = np.hypot(Xs[:, 0], Xs[:, 1]) > R
        X, N = np.concatenate([X[keep], Xs[ks]]), np.concatenate([N[keep], Ns[ks]])
        dS = np.concatenate([dS[keep], np.full(int(ks.sum()), 4 * math.pi * rs * rs / len(s))])
        inside = (np.hypot(x, y) < R) | ((x - off) ** 2 + y ** 2 + (z - 0.5 * L) ** 2 < rs * rs)
        outlet = (2, 1, (0.0, 0.0, L))
    else:
        arc = 0.5 * math.pi * rc
        total = 2 * leg + arc
        s, t = _strata(lay, max(8, int(round(total / d))), th_n)
        s, th = s * total, 2 * math.pi * t
        a = np.clip((s - leg) / rc, 0.0, 0.5 * math.pi)
        nrm = np.stack([-np.cos(a), 0 * a, np.sin(a)], 1)                # away from the bend's centre
        cen = np.stack([rc - rc * np.cos(a), 0 * a, leg + rc * np.sin(a)], 1)
        cen[:, 2] += np.minimum(s - leg, 0.0)
        cen[:, 0] += np.maximum(s - leg - arc, 0.0)
        N = np.cos(th)[:, None] * nrm + np.sin(th)[:, None] * np.array([0.0, 1.0, 0.0])
        X = cen + R * N
        bent = (s > leg) & (s < leg + arc)
        dS = np.where(bent, 1 + R / rc * np.cos(th), 1.0) * total * 2 * math.pi * R / len(s)
        rr = np.hypot(x - rc, z - leg)
        inside = ((z < leg) & (np.hypot(x, y) < R)) | ((z >= leg) & (x <= rc) & (np.hypot(rr - rc, y) < R)) | (
            (x > rc) & (np.hypot(z - leg - rc, y) < R))
        outlet = (0, 1, (rc + leg, 0.0, leg + rc))
    # the grid follows the coarse cells that hold points: the seed moves no point to another one
    X2 = X + 0.1 * d * rng.uniform(-1, 1, X.shape)
    X2[:, 2] = np.clip(X2[:, 2], 0.0, ext[2])
    cell = [np.floor((P - np.array(lo)) / np.array(hc)) for P in (X, X2)]
    X = np.where((cell[0] == cell[1]).all(1, keepdims=True), X2, X)
    peak = rng.uniform(0.85, 1.0)
    puls = rng.uniform(0.2, 0.4)
    pin = case["inlet"] == "pressure"
    f = 16.0 * case["nu"] * L / R ** 2 if pin else 1.0      # the pressure of a Poiseuille flow with this peak
    ports = [dict(axis=2, side=0, center=(0.0, 0.0, 0.0), radius=R, kind="pinlet" if pin else "inlet", a0=f * peak,
                  a=(), b=(f * peak * puls,), period=1.0),
             dict(axis=outlet[0], side=outlet[1], center=outlet[2], radius=R, kind="outlet", a0=0.0, a=(), b=(),
                  period=1.0)]
    return dict(origin=tuple(lo), extent=tuple(ext), n=tuple(int(v) for v in n), max_level=int(case["levels"]),
                refine_band=2, reduce_band=-1 if kind == "tube" and case["levels"] == 0 else 2, nu=float(case["nu"]),
                rho=1.0, dt=case["cfl"] * hf, ports=ports, X=np.ascontiguousarray(X), dS=dS, UB=np.zeros_like(X),
                inside=inside.astype(np.uint8), viscous=case["viscous"], normals=N, hf=hf)


def _members(case, seed):
    """The problems of a case: one, or the members of a batch (shapes, depths and sizes in turn)."""
    rng = np.random.default_rng(seed)
    if case["call"] != "batch":
        return [_vessel(case, rng)]
    got = []
    for k in range(case["members"]):
        lev = (0, 1, case["levels"], 1)[k % 4]
        n = max(8, int(round(case["n"] * (1.4, 0.9, 0.65, 0.8)[k % 4])))
        got.append(_vessel(dict(case, kind=("tube", "sac", "bend")[k % 3], levels=lev, n=n,
                                z_cells=max(8, int(round(case["z_cells"] * n / case["n"]))),
                                nu=max(case["nu"], 0.8 / n)), rng))
    return got


_FRAMES = 16


def _frames(v):
    """The wall of a moving tube: radial pulsation of 0.3 finest cells, with its velocity."""
    w = 2 * math.pi / (_FRAMES * v["dt"])
    amp = 0.3 * v["hf"]
    ph = 2 * math.pi * (np.arange(_FRAMES) + 1) / _FRAMES
    X = v["X"][None] + amp * np.sin(ph)[:, None, None] * v["normals"][None]
    U = amp * w * np.cos(ph)[:, None, None] * v["normals"][None]
    X[..., 2] = np.clip(X[..., 2], 0.0, v["extent"][2])
    return X, U


def _smooth_flow(v, x):
    """A developed flow at the points x: Poiseuille with a swirl and a pulsating part."""
    r2 = (x[..., 0] ** 2 + x[..., 1] ** 2) / 0.25
    k = 2 * math.pi / v["extent"][2]
    w = (v["ports"][0]["a0"] + 0.1 * np.sin(k * x[..., 2])) * (1 - r2)
    return np.stack([-0.3 * x[..., 1] * (1 - r2), 0.3 * x[..., 0] * (1 - r2), w], -1)


# ---------------------------------------------------------------------------
# What is measured
# ---------------------------------------------------------------------------
def prepare(case, seed):
    vs = _members(case, seed)
    if case["call"] == "batch":
        grids = [IBGrid(v, precision=case["precision"], deferred=True) for v in vs]
        state = {"batch": IBBatch(grids)}
    else:
        grids = [IBGrid(vs[0], precision=case["precision"])]
        state = {}
    state.update(call=case["call"], grids=grids, normals=vs[0]["normals"], pass_=0)
    if case["call"] == "wss":
        g, v = grids[0], vs[0]
        q = g.ib_fields_get("NODE_Q")
        hf = np.array(v["extent"]) / (np.array(v["n"]) << v["max_level"])
        g.ib_fields_set("U", _smooth_flow(v, np.array(v["origin"]) + q * hf))
        return state
    if case["call"] == "move":
        state["X"], state["UB"] = (torch.from_numpy(a).cuda() for a in _frames(vs[0]))
    state["out"] = []
    for g in grids:
        n = g.ib_grid_info()["n_nodes"]
        state["out"].append((torch.empty((n, 3), dtype=torch.float64, device="cuda"),
                             torch.empty((n,), dtype=torch.float64, device="cuda")))
    return state


def run(state):
    if state["call"] == "wss":
        w, grad = state["grids"][0].ib_wss(state["normals"], with_grad=True)
        return {"wss": w, "grad": grad}
    res = {}
    if state["call"] == "batch":
        res["status"] = state["batch"].step(1)
    else:
        if state["call"] == "move":
            k = state["pass_"] % _FRAMES
            state["pass_"] += 1
            state["grids"][0].ib_set_points(state["X"][k], state["UB"][k])
        state["grids"][0].ipcs_step(1)
    for i, (g, (u, p)) in enumerate(zip(state["grids"], state["out"])):
        res["U%d" % i] = g.ib_fields_get("U", out=u)
        res["P%d" % i] = g.ib_fields_get("P", out=p)
    return res


def work(case):
    nodes = points = 0
    for v in _members(case, 0):
        level, active = _level_map(v)
        nodes += int((8 ** level[active].to(torch.int64)).sum())     # a leaf cell has about one node
        points += len(v["X"])
    if case["call"] == "wss":
        # the nodes within reach of a point, about a half ball of 3.5 spacings; the moment matrix and the derivatives
        near = 0.5 * 4 / 3 * math.pi * 3.5 ** 3
        return {"bytes": points * (8.0 * (3 + 3 + 3 + 1 + 9) + 24 * case["spacing"] ** 2 * 4),
                "flops": points * near * 160.0}
    # the state (u, p) in and out and read back, the nodes' cell masks; Eq. 9, Eq. 12 and the correction applied once
    return {"bytes": nodes * (32.0 * 3 + 2) + points * (24.0 * 4 + 64 * 8),
            "flops": nodes * (3 * 2 * 15 * 2 + 2 * 7 + 500.0) + points * 64 * 6 * 2.0}


# ---------------------------------------------------------------------------
# The same in 64 bits with torch alone: assembled matrices, plain CG, on the
# first step from rest (no convection yet, so the momentum matrix is symmetric)
# ---------------------------------------------------------------------------
_PERMS = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))
_EXACT_CELLS = 4_500_000


def _grow(m):
    return torch.nn.functional.max_pool3d(m[None, None].float(), 3, 1, 1)[0, 0]


def _level_map(v):
    """Refinement level and activity of the coarse cells [z][y][x]: levels by Chebyshev distance to a cell that holds a
    point, one less per band of two cells, 2:1 balanced; active where inside or within two cells of such a cell."""
    n, L = np.array(v["n"]), v["max_level"]
    c = np.floor((v["X"] - np.array(v["origin"])) / (np.array(v["extent"]) / n)).astype(np.int64)
    m = torch.zeros((n[2], n[1], n[0]))
    m[c[:, 2], c[:, 1], c[:, 0]] = 1
    level, reach = torch.zeros(m.shape, dtype=torch.int32), m
    active = torch.from_numpy(np.asarray(v["inside"])).bool() if v["reduce_band"] >= 0 else torch.ones_like(m).bool()
    for d in range(0, 2 * L + 3):
        if d:
            reach = _grow(reach)
        k = 0 if d <= 2 else -(-(d - 2) // 2)
        level = torch.maximum(level, ((L - k) * (reach > 0)).to(torch.int32).clamp(min=0))
        if d == v["reduce_band"]:
            active = active | (reach > 0)
    for _ in range(L + 1):
        level = torch.maximum(level, (_grow(level).to(torch.int32) - 1).clamp(min=0))
    return level, active


class _Mesh:
    def __init__(self, v):
        dev = "cuda"
        self.v, L = v, v["max_level"]
        n = torch.tensor(v["n"], device=dev)
        self.nf = n * (1 << L)
        self.x0 = torch.tensor(v["origin"], dtype=torch.float64, device=dev)
        self.hf = torch.tensor(v["extent"], dtype=torch.float64, device=dev) / self.nf.double()
        level, active = (t.to(dev) for t in _level_map(v))
        corner, size = [], []
        for l in range(L + 1):
            z, y, x = torch.nonzero(active & (level == l), as_tuple=True)
            m = 1 << l
            s = torch.arange(m, device=dev)
            sub = torch.stack(torch.meshgrid(s, s, s, indexing="ij"), -1).reshape(-1, 3)
            c = (torch.stack([x, y, z], 1)[:, None] * (1 << L) + (1 << (L - l)) * sub[None]).reshape(-1, 3)
            corner.append(c)
            size.append(torch.full((len(c),), 1 << (L - l), device=dev))
        self.corner, self.size = torch.cat(corner), torch.cat(size)
        bits = torch.tensor([[b & 1, b >> 1 & 1, b >> 2] for b in range(8)], device=dev)
        self.keys, inv = torch.unique(self.key(self.corner[:, None] + self.size[:, None, None] * bits[None]),
                                      return_inverse=True)
        self.cells = inv.reshape(-1, 8)
        sx, sy = self.nf[0] + 1, self.nf[1] + 1
        self.q = torch.stack([self.keys % sx, self.keys // sx % sy, self.keys // (sx * sy)], 1)
        self.x = self.x0 + self.q * self.hf
        self.N = len(self.keys)
        # hanging nodes: midpoints of a larger cell's edges and face diagonals
        self.hang = torch.zeros(self.N, dtype=torch.bool, device=dev)
        self.par = torch.zeros((self.N, 2), dtype=torch.int64, device=dev)
        big = self.size >= 2
        for a in range(8):
            for b in range(8):
                d = a ^ b
                if a & b != a or d == 0 or d == 7:
                    continue                       # b = a plus one or two axes: cube edges and Kuhn face diagonals
                ca, cb = (self.corner[big] + self.size[big, None] * bits[k] for k in (a, b))
                i = self.find((ca + cb) // 2)
                ok = i >= 0
                self.hang[i[ok]] = True
                self.par[i[ok]] = torch.stack([self.find(ca[ok]), self.find(cb[ok])], 1)
        # boundary of the active cells, ports
        bnd = torch.zeros(self.N, dtype=torch.bool, device=dev)
        for k in range(8):
            c = torch.div(2 * self.q + 2 * bits[k] - 1, 2 << L, rounding_mode="floor")
            inb = ((c >= 0) & (c < n)).all(1)
            c = torch.minimum(c.clamp(min=0), n - 1)
            bnd |= ~(inb & active[c[:, 2], c[:, 1], c[:, 0]])
        self.port, taken = [], torch.zeros_like(bnd)
        for p in v["ports"]:
            o = [a for a in range(3) if a != p["axis"]]
            plane = 0 if p["side"] == 0 else self.nf[p["axis"]]
            d0, d1 = (self.x[:, a] - p["center"][a] for a in o)
            r2 = d0 * d0 + d1 * d1
            sel = (self.q[:, p["axis"]] == plane) & bnd & (r2 <= p["radius"] ** 2) & ~taken
            taken |= sel
            self.port.append((sel & ~self.hang, r2))
        free_port = torch.zeros_like(bnd)
        for p, (sel, _) in zip(v["ports"], self.port):
            if p["kind"] != "inlet":
                free_port |= sel
        self.pdir = free_port
        self.vdir = bnd & ~free_port & ~self.hang
        # P: all nodes from the free ones (a hanging node is the mean of its parents)
        i = torch.arange(self.N, device=dev)
        h = i[self.hang]
        self.P = _csr(torch.cat([i[~self.hang], h, h]), torch.cat([i[~self.hang], self.par[h, 0], self.par[h, 1]]),
                      torch.cat([torch.ones(self.N - len(h), dtype=torch.float64, device=dev),
                                 torch.full((2 * len(h),), 0.5, dtype=torch.float64, device=dev)]), self.N)
        self.PT = _csr(torch.cat([i[~self.hang], self.par[h, 0], self.par[h, 1]]), torch.cat([i[~self.hang], h, h]),
                       torch.cat([torch.ones(self.N - len(h), dtype=torch.float64, device=dev),
                                  torch.full((2 * len(h),), 0.5, dtype=torch.float64, device=dev)]), self.N)

    def key(self, q):
        return (q[..., 2] * (self.nf[1] + 1) + q[..., 1]) * (self.nf[0] + 1) + q[..., 0]

    def find(self, q):
        k = self.key(q)
        i = torch.searchsorted(self.keys, k).clamp(max=self.N - 1)
        ok = (self.keys[i] == k) & ((q >= 0) & (q <= self.nf)).all(-1)
        return torch.where(ok, i, torch.full_like(i, -1))

    def assemble(self, form):
        """The matrix of the cell form(spacing) -> 8x8, summed over the leaf cells."""
        A = None
        for s in torch.unique(self.size).tolist():
            E = form((self.hf * s).tolist()).cuda()
            c = self.cells[self.size == s]
            nz = torch.nonzero(E.abs() > 1e-14 * E.abs().max())
            for part in c.split(2_000_000):
                r = part[:, nz[:, 0]].reshape(-1)
                k = part[:, nz[:, 1]].reshape(-1)
                w = E[nz[:, 0], nz[:, 1]].expand(len(part), -1).reshape(-1)
                B = torch.sparse_coo_tensor(torch.stack([r, k]), w, (self.N, self.N)).coalesce()
                A = B if A is None else (A + B).coalesce()
        return A.to_sparse_csr()


def _csr(r, c, w, n, m=None):
    return torch.sparse_coo_tensor(torch.stack([r, c]), w, (n, m or n)).coalesce().to_sparse_csr()


def _tet(h, perm):
    """Corners of one Kuhn tetrahedron and the gradients of its barycentric functions."""
    c = [0, 1 << perm[0], (1 << perm[0]) | (1 << perm[1]), 7]
    g = torch.zeros((4, 3), dtype=torch.float64)
    for k, a in enumerate(perm):
        g[k, a] -= 1 / h[a]
        g[k + 1, a] += 1 / h[a]
    return c, g


def _form(h, entry):
    E = torch.zeros((8, 8), dtype=torch.float64)
    vol = h[0] * h[1] * h[2] / 6
    for perm in _PERMS:
        c, g = _tet(h, perm)
        for i in range(4):
            for j in range(4):
                E[c[i], c[j]] += entry(vol, g, i, j)
    return E


def _cg(A, b, diag, free, x, iters=20000):
    """A x = b on the free rows, x given on the others; columns side by side; to the end of 64 bits."""
    fr = free[:, None].double()
    minv = fr / torch.where(free, diag, torch.ones_like(diag))[:, None]
    r = fr * (b - A(x))
    ref = torch.maximum((fr * b).norm(dim=0), r.norm(dim=0)).clamp(min=1e-300)
    z = minv * r
    p, rz = z.clone(), (r * z).sum(0)
    for k in range(iters):
        q = fr * A(p)
        pq = (p * q).sum(0)
        al = torch.where(pq > 0, rz / pq.clamp(min=1e-300), torch.zeros_like(rz))
        x = x + al * p
        r = r - al * q
        z = minv * r
        new = (r * z).sum(0)
        p = z + torch.where(rz > 0, new / rz.clamp(min=1e-300), torch.zeros_like(rz)) * p
        rz = new
        if k % 16 == 15 and bool((r.norm(dim=0) <= 2e-15 * ref).all()):
            break
    return x


def _diag(A):
    coo = A.to_sparse_coo().coalesce()
    i = coo.indices()
    on = i[0] == i[1]
    d = torch.zeros(A.shape[0], dtype=torch.float64, device="cuda")
    d[i[0][on]] = coo.values()[on]
    return d


def _kernel(r):
    r = r.abs()
    a = (3 - 2 * r + (1 + 4 * r - 4 * r * r).clamp(min=0).sqrt()) / 8
    b = (5 - 2 * r - (-7 + 12 * r - 4 * r * r).clamp(min=0).sqrt()) / 8
    return torch.where(r <= 1, a, torch.where(r <= 2, b, torch.zeros_like(r)))


def _first_step(v, X, UB):
    """u and p after one step from rest with the wall points at X."""
    m = _Mesh(v)
    dt, nu = v["dt"], v["nu"]
    M = m.assemble(lambda h: _form(h, lambda vol, g, i, j: vol * (2 if i == j else 1) / 20))
    K = m.assemble(lambda h: _form(h, lambda vol, g, i, j: vol * float(g[i] @ g[j])))
    G = [m.assemble(lambda h, a=a: _form(h, lambda vol, g, i, j: vol / 4 * float(g[j, a]))) for a in range(3)]

    def solve(A, b, dirichlet, x):
        op = lambda y: m.PT @ (A @ (m.P @ y))  # noqa: E731
        # the condensed diagonal: sum_ij P_ik A_ij P_jk = A_kk + sums over hanging children
        d = _diag(A)
        hid = torch.nonzero(m.hang)[:, 0]
        c = A.to_sparse_coo().coalesce()
        d = d.clone()
        for s in (0, 1):
            d.index_add_(0, m.par[hid, s], 0.25 * d[hid])
        # the off-diagonal couplings of a child with its parent and with the parent's other children
        i, w = c.indices(), c.values()
        sel = (m.hang[i[0]] | m.hang[i[1]]) & (i[0] != i[1])
        ii, jj, w = i[0][sel], i[1][sel], w[sel]
        one = torch.arange(m.N, device="cuda")
        pi = torch.where(m.hang[:, None], m.par, torch.stack([one, torch.full_like(one, -1)], 1))
        wi = torch.where(m.hang, 0.5, 1.0).double()
        for s in (0, 1):
            for t in (0, 1):
                a, b_ = pi[ii, s], pi[jj, t]
                eq = (a == b_) & (a >= 0)
                d.index_add_(0, a[eq], (w * wi[ii] * wi[jj])[eq])
        free = ~dirichlet & ~m.hang
        return m.P @ _cg(op, b, d, free, torch.where(m.hang[:, None], torch.zeros_like(x), x))

    def wave(p):
        s = p["a0"]
        for k, b in enumerate(p["b"], 1):
            s += b * math.sin(2 * math.pi * k * dt / p["period"])
        return s

    g = torch.zeros((m.N, 3), dtype=torch.float64, device="cuda")
    gp = torch.zeros((m.N, 1), dtype=torch.float64, device="cuda")
    for p, (sel, r2) in zip(v["ports"], m.port):
        if p["kind"] == "inlet":
            g[:, p["axis"]] = torch.where(sel, wave(p) * (1 - r2 / p["radius"] ** 2), g[:, p["axis"]])
        elif p["kind"] == "pinlet":
            gp[:, 0] = torch.where(sel, torch.full_like(r2, wave(p)), gp[:, 0])
    zero = torch.zeros((m.N, 3), dtype=torch.float64, device="cuda")
    ut = zero if float(g.abs().max()) == 0 else solve((M + (dt * nu) * K), zero, m.vdir, g)
    # force system on the free nodes around the points
    X, UB = torch.from_numpy(X).cuda(), torch.from_numpy(UB).cuda()
    o = torch.floor((X - m.x0) / m.hf).long() - 1
    off = torch.tensor([[a & 3, a >> 2 & 3, a >> 4] for a in range(64)], device="cuda")
    q = o[:, None] + off[None]
    w = _kernel((m.x0 + q * m.hf - X[:, None]) / m.hf).prod(-1)
    node = m.find(q)
    has = node >= 0
    row = torch.arange(len(X), device="cuda")[:, None].expand(-1, 64)
    W = _csr(row[has], node[has], w[has], len(X), m.N)
    fr = has & (~m.vdir & ~m.hang)[node.clamp(min=0)]
    Wf = _csr(row[fr], node[fr], w[fr], len(X), m.N)
    WfT = _csr(node[fr], row[fr], w[fr], m.N, len(X))
    h3 = float(m.hf.prod())
    bf = UB - W @ ut
    u = ut
    if float(bf.abs().max()) > 0:
        sc = dt / v["rho"] / h3
        d = sc * torch.zeros(len(X), dtype=torch.float64, device="cuda").index_add_(0, row[fr], w[fr] ** 2)
        F = _cg(lambda y: sc * (Wf @ (WfT @ y)), bf, d, torch.ones(len(X), dtype=torch.bool, device="cuda"),
                torch.zeros_like(bf), 6000)
        u = ut + sc * (WfT @ F)
    div = sum(G[a] @ u[:, a:a + 1] for a in range(3))
    phi = solve(K, m.PT @ (-div / dt), m.pdir, gp)
    b = torch.cat([m.PT @ (M @ u[:, a:a + 1] - dt * (G[a] @ phi)) for a in range(3)], 1)
    return solve(M, b, m.vdir, g), phi[:, 0]


def _wall_shear(v):
    """Wall shear stress and velocity gradient at the points by second-order DC-PSE operators: nodes of the finest cells
    within 3.5 of the largest finest spacing on the fluid side, Gaussian weights, exact for polynomials of degree 2."""
    m = _Mesh(v)
    u = torch.from_numpy(_smooth_flow(v, m.x.cpu().numpy())).cuda()
    u = m.P @ u
    fine = torch.zeros(m.N, dtype=torch.bool, device="cuda")
    fine[m.cells[m.size == 1].reshape(-1)] = True
    X, nrm = torch.from_numpy(v["X"]).cuda(), torch.from_numpy(v["normals"]).cuda()
    e = float(m.hf.max())
    rad = [int(math.ceil(3.5 * e / float(h))) for h in m.hf]
    rng_ = [torch.arange(-r, r + 2, device="cuda") for r in rad]
    off = torch.stack(torch.meshgrid(*rng_, indexing="ij"), -1).reshape(-1, 3)
    ws, gs = [], []
    for s in range(0, len(X), 2048):
        x, n = X[s:s + 2048], nrm[s:s + 2048]
        q = torch.floor((x - m.x0) / m.hf).long()[:, None] + off[None]
        i = m.find(q)
        d = (m.x0 + q * m.hf) - x[:, None]
        r2 = d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1] + d[..., 2] * d[..., 2]
        dn = d[..., 0] * n[:, None, 0] + d[..., 1] * n[:, None, 1] + d[..., 2] * n[:, None, 2]
        sel = (i >= 0) & (r2 <= (3.5 * e) ** 2) & (dn < 0) & fine[i.clamp(min=0)]
        z = d / e
        mono = torch.stack([z[..., 0], z[..., 1], z[..., 2], z[..., 0] ** 2, z[..., 0] * z[..., 1],
                            z[..., 0] * z[..., 2], z[..., 1] ** 2, z[..., 1] * z[..., 2], z[..., 2] ** 2], -1)
        wt = torch.where(sel, torch.exp(-(z * z).sum(-1)), torch.zeros_like(r2))
        A = torch.einsum("pq,pqi,pqj->pij", wt, mono, mono)
        rhs = torch.eye(9, dtype=torch.float64, device="cuda")[:, :3].expand(len(x), 9, 3)
        eta = torch.einsum("pqi,pij->pqj", mono, torch.linalg.solve(A, rhs)) * wt[..., None]
        gs.append(torch.einsum("pqi,pqj->pij", u[i.clamp(min=0)], eta) / e)
        t = v["nu"] * torch.einsum("pij,pj->pi", gs[-1] + gs[-1].transpose(1, 2), n)
        ws.append((t - (t * n).sum(1, keepdim=True) * n).norm(dim=1))
    return {"wss": torch.cat(ws), "grad": torch.cat(gs)}


def exact(case, seed):
    vs = _members(case, seed)
    cells = 0
    for v in vs:
        level, active = _level_map(v)
        cells += int((8 ** level[active].to(torch.int64)).sum())
    if cells > _EXACT_CELLS:
        return None                                # assembling and solving would take too long
    if case["call"] == "wss":
        return _wall_shear(vs[0])
    res = {"status": None} if case["call"] == "batch" else {}
    for i, v in enumerate(vs):
        X, UB = v["X"], v["UB"]
        if case["call"] == "move":
            fx, fu = _frames(v)
            X, UB = np.ascontiguousarray(fx[0]), np.ascontiguousarray(fu[0])
        res["U%d" % i], res["P%d" % i] = _first_step(v, X, UB)
    return res
