"""Workloads by which the speed of the S_N step is measured.

A pass is what a user's time loop does between two looks at the solution: advance
the solver (or the batch) by a few steps with `step`, read the QoIs, and take the
device view of the state (psi and phi, rt_device_state) or, for a batch, the QoIs
of all its members. Geometries, grids, ordinate sets and schemes are those of the
benchmarks: the lattice on Cartesian grids (70^2 to 1400^2 cells), the enclosure
on jittered triangle meshes (130^2 to 1300^2 split squares), the product rules of
64 to 512 ordinates, the tessellation rule, first order with Euler and second
order with Heun, FP32 and BF16 storage.

States are positive and vary in space, angle and from cell to cell, as in the
middle of a solve; cross-sections are drawn over the ranges of the parameter
sweeps. Problems run towards an end time that is never reached, so that a solver
can be advanced as often as wanted.
"""
from dataclasses import replace
from functools import lru_cache

import numpy as np
import torch

import sn_inputs as si
from paper_2505_17284_gb300 import rt

MANY_STEPS = 10_000_000          # t_end in units of dt
LARGEST = 1400 * 1400 * 512      # cells x ordinates x steps of the largest listed case
BATCH_SPIN_UP = 64               # steps a batch has made (from psi = 0) before the first pass
PRODUCT = {64: (4, 16), 128: (8, 16), 256: (8, 32), 512: (16, 32)}   # polar x azimuthal points


def _lattice(name, n, M, order, heun, storage, steps):
    return {"name": name, "kind": "lattice", "n": n, "M": M, "order": order, "heun": heun, "storage": storage,
            "steps": steps}


def _enclosure(name, n, M, order, heun, storage, steps):
    return {"name": name, "kind": "enclosure", "n": n, "M": M, "order": order, "heun": heun, "storage": storage,
            "steps": steps}


def listed():
    return [
        # the benchmark's plain configuration, one step at a time: the smallest call
        _lattice("lattice70_m64_o1_euler", 70, 64, 1, False, "fp32", 1),
        # a small solve of a parameter sweep, in stretches of 32 steps
        _lattice("lattice140_m128_o2_heun", 140, 128, 2, True, "fp32", 32),
        # a medium solve with 256 ordinates
        _lattice("lattice280_m256_o2_heun", 280, 256, 2, True, "fp32", 8),
        # a grid that no tile divides, with 100 ordinates of the tessellation rule (padded to 128 in memory)
        _lattice("lattice531_tess5_o2_heun", 531, 100, 2, True, "fp32", 4),
        # the largest grid of the serving stream with 484 tessellation ordinates (121 per quadrant)
        _lattice("lattice700_tess11_o2_heun", 700, 484, 2, True, "fp32", 2),
        # the lattice at production size: the headline workload, then its BF16 storage, then first order
        _lattice("lattice1400_m512_o2_heun", 1400, 512, 2, True, "fp32", 1),
        _lattice("lattice1400_m512_o2_heun_bf16", 1400, 512, 2, True, "bf16", 1),
        _lattice("lattice1400_m512_o1_euler", 1400, 512, 1, False, "fp32", 1),
        # the smallest enclosure of the serving stream
        _enclosure("enclosure130_m64_o1_euler", 130, 64, 1, False, "fp32", 16),
        # the enclosure at production size, first order
        _enclosure("enclosure1300_m256_o1_euler", 1300, 256, 1, False, "fp32", 1),
        # the paper's second-order scheme on triangles
        _enclosure("enclosure650_m256_o2_heun", 650, 256, 2, True, "fp32", 1),
        # a batched parameter sweep over small lattices (70^2 and 140^2 cells; 64, 128 and 256 ordinates)
        {"name": "sweep24_o2_heun", "kind": "sweep", "members": 24, "n": 70, "n_large": 140, "order": 2, "heun": True,
         "storage": "fp32", "steps": 16},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(lo * (hi / lo) ** rng.random()))

    kind = rng.choice(["lattice", "lattice", "lattice", "enclosure", "enclosure", "sweep"])
    storage = rng.choice(["fp32", "fp32", "bf16"])
    if kind == "sweep":
        n = rng.randint(50, 90)
        return {"kind": "sweep", "members": rng.randint(8, 32), "n": n, "n_large": rng.randint(n + 20, 160), "order": 2,
                "heun": True, "storage": "fp32", "steps": rng.choice([4, 8, 16])}
    heun = rng.random() < 0.6
    order = 2 if heun else 1
    if kind == "lattice":
        M = rng.choice([64, 128, 256, 512, 100, 256, 484])
        n = log_int(70, 1400)
    else:
        M = rng.choice([64, 128, 256])
        n = log_int(60, 900 if order == 1 else 650)
    cells = n * n * (2 if kind == "enclosure" else 1)
    weight = 4 if kind == "enclosure" and order == 2 else 1
    most = max(1, LARGEST // (4 * cells * M * weight))
    return {"kind": kind, "n": n, "M": M, "order": order, "heun": heun, "storage": storage,
            "steps": min(most, rng.choice([1, 2, 4, 16, 32]))}


# ---------------------------------------------------------------------------- inputs
@lru_cache(maxsize=None)
def _quad(M):
    if M in PRODUCT:
        return rt.rt_quad_product(*PRODUCT[M])
    N = int(round((M / 4) ** 0.5))
    assert 4 * N * N == M
    return rt.rt_quad_tessellation(N)


@lru_cache(maxsize=4)
def _geometry(kind, n):
    return si.lattice_problem(n) if kind == "lattice" else si.enclosure_problem(n, jitter=0.2, seed=0)


def _problem(kind, n, rng):
    """The geometry with cross-sections drawn over the sweeps' ranges."""
    p = _geometry(kind, n)
    if kind == "lattice":
        sa, ss, q = si.lattice_materials_table(rng.uniform(5, 15), *[rng.uniform(0.5, 1.5)] * 2)
    else:
        sa, ss, q = si.enclosure_materials_table(rng.uniform(60, 120))
    return replace(p, materials=replace(p.materials, sigma_a=sa, sigma_s=ss, Q=q))


@lru_cache(maxsize=4)
def _mesh(n):
    """Metrics of the enclosure's mesh in FP64 and the order in which a solver keeps
    its cells (Morton order of the centroids, ties by index)."""
    m = _geometry("enclosure", n).mesh
    P = m.vertices[m.triangles]
    Pn = np.roll(P, -1, axis=1)
    a, b, c = P[:, 0], P[:, 1], P[:, 2]
    area = 0.5 * ((b[:, 0] - a[:, 0]) * (c[:, 1] - a[:, 1]) - (b[:, 1] - a[:, 1]) * (c[:, 0] - a[:, 0]))
    nl = np.stack([Pn[..., 1] - P[..., 1], P[..., 0] - Pn[..., 0]], axis=2)
    cen = P.mean(axis=1)
    mid = 0.5 * (P + Pn)
    tri = m.triangles.astype(np.int64)
    p, q = tri.ravel(), np.roll(tri, -1, axis=1).ravel()
    key = np.minimum(p, q) * (tri.max() + 1) + np.maximum(p, q)
    by = np.argsort(key, kind="stable")
    twin = np.full(key.size, -1, dtype=np.int64)
    same = np.nonzero(key[by][1:] == key[by][:-1])[0]
    twin[by[same]], twin[by[same + 1]] = by[same + 1], by[same]
    nbr = np.where(twin >= 0, twin // 3, -1).reshape(-1, 3)
    x0, y0, x1, y1 = m.box
    far = np.stack([np.abs(mid[..., 0] - x0), np.abs(mid[..., 0] - x1), np.abs(mid[..., 1] - y0), np.abs(mid[..., 1] - y1)])
    side = np.where(nbr < 0, np.argmin(far, axis=0), -1)
    cx = (m.vertices[tri[:, 0], 0] + m.vertices[tri[:, 1], 0] + m.vertices[tri[:, 2], 0]) / 3.0
    cy = (m.vertices[tri[:, 0], 1] + m.vertices[tri[:, 1], 1] + m.vertices[tri[:, 2], 1]) / 3.0

    def grid(v):
        u = ((v - v.min()) * (65535.0 / (v.max() - v.min()))).astype(np.uint64)
        for s, k in ((8, 0x00FF00FF), (4, 0x0F0F0F0F), (2, 0x33333333), (1, 0x55555555)):
            u = (u | (u << np.uint64(s))) & np.uint64(k)
        return u

    perm = np.argsort(grid(cx) | (grid(cy) << np.uint64(1)), kind="stable")
    dt = 0.9 * float(np.min(2.0 * area / np.linalg.norm(nl, axis=2).sum(axis=1)))
    return {"area": area, "nl": nl, "cen": cen, "mid": mid, "nbr": nbr, "side": side, "perm": perm, "dt": dt}


def _setup(case, seed):
    rng = np.random.default_rng(seed)
    p = _problem(case["kind"], case["n"], rng)
    quad = _quad(case["M"])
    dt = 0.5 * p.mesh.dx if case["kind"] == "lattice" else _mesh(case["n"])["dt"]
    return p, quad, dt


@lru_cache(maxsize=4)
def _centres(kind, n):
    if kind == "lattice":
        x, y = _geometry(kind, n).mesh.centres()
    else:
        m = _mesh(n)
        x, y = m["cen"][m["perm"]].T
    return torch.as_tensor(np.stack([x, y]), dtype=torch.float32, device="cuda")


def _fill(psi, phi, case, seed, w):
    """A positive state [cell][ordinate] in the solver's order of the cells: a bump in
    space times a profile in angle times 10 % of noise, and its scalar flux."""
    rng = np.random.default_rng(seed + 1)
    g = torch.Generator(device="cuda").manual_seed(seed)
    x, y = _centres(case["kind"], case["n"])
    L = 7.0 if case["kind"] == "lattice" else 1.3
    cx, cy = rng.uniform(0.3 * L, 0.7 * L, size=2)
    bump = 0.05 + torch.exp(((x - cx) ** 2 + (y - cy) ** 2) / (-2 * (0.2 * L) ** 2))
    profile = torch.as_tensor(rng.uniform(0.5, 1.5, size=psi.shape[1]), dtype=torch.float32, device="cuda")
    weights = torch.as_tensor(w, dtype=torch.float32, device="cuda")
    rows = max(1, (1 << 28) // psi.shape[1])
    for i in range(0, psi.shape[0], rows):
        u = torch.empty((min(rows, psi.shape[0] - i), psi.shape[1]), dtype=torch.float32, device="cuda")
        u.uniform_(0.9, 1.1, generator=g).mul_(bump[i:i + rows, None]).mul_(profile)
        psi[i:i + rows] = u
        if phi is not None:
            phi[i:i + rows] = psi[i:i + rows].float() @ weights


# ---------------------------------------------------------------------------- a solver and its device view
class _Array:
    """Device memory of a solver, which stays alive as long as a tensor on it does."""

    def __init__(self, solver, ptr, shape, typestr):
        self.solver = solver
        self.__cuda_array_interface__ = {"data": (ptr, False), "shape": shape, "typestr": typestr, "version": 3}


def _view(state):
    """psi [cell][ordinate] and phi [cell] of the current state, without a copy. A
    regrouped solver keeps each of the four quadrants padded: [cell][quadrant][ordinate]."""
    s = state["solver"]
    p, f, storage = rt.rt_device_state(s.h)
    if (p, f) not in state["views"]:
        rows = int(s.info.M_pad)
        psi = torch.as_tensor(_Array(s, p, (s.n_cells, rows), "<f4" if storage == rt.RT_FP32 else "<i2"), device="cuda")
        if storage == rt.RT_BF16:
            psi = psi.view(torch.bfloat16)
        psi = psi.view(s.n_cells, 4, rows // 4)[:, :, :s.M // 4] if s.info.regrouped else psi[:, :s.M]
        state["views"][p, f] = psi, torch.as_tensor(_Array(s, f, (s.n_cells,), "<f4"), device="cuda")
    return state["views"][p, f]


def _now(q):
    """QoIs of a state as plain numbers."""
    return {"abs": [float(v) for v in q["abs_now"]], "mass": float(q["mass"]), "outflow": float(q["outflow_now"]),
            "box_out": [float(v) for v in q["box_out_now"]]}


def _members(case, seed):
    """(grid, ordinates, absorption, scattering) of a sweep's members."""
    rng = np.random.default_rng(seed)
    sizes = [(n, M) for M in (64, 128, 256) for n in (case["n"], case["n_large"])]
    return [(*sizes[i % 6], rng.uniform(5, 15), rng.uniform(0.5, 1.5)) for i in range(case["members"])]


def _member_problem(n, sa, ss):
    p = _geometry("lattice", n)
    t = si.lattice_materials_table(sa, ss, ss)
    m = replace(p.materials, sigma_a=t[0], sigma_s=t[1], Q=t[2])
    return replace(p, materials=m, t_end=0.5 * p.mesh.dx * MANY_STEPS)


def prepare(case, seed):
    storage = rt.RT_BF16 if case["storage"] == "bf16" else rt.RT_FP32
    integrator = rt.RT_HEUN if case["heun"] else rt.RT_EULER
    if case["kind"] == "sweep":
        b = rt.Batch([], [], capacity=case["members"], storage=storage)
        for n, M, sa, ss in _members(case, seed):
            p = _member_problem(n, sa, ss)
            b.add(p, _quad(M), order=case["order"], integrator=integrator, dt=0.5 * p.mesh.dx)
        b.step(BATCH_SPIN_UP)
        return {"batch": b, "members": case["members"], "steps": case["steps"]}
    p, quad, dt = _setup(case, seed)
    s = rt.Solver(p, quad, order=case["order"], integrator=integrator, storage=storage, dt=dt, t_end=dt * MANY_STEPS)
    state = {"solver": s, "steps": case["steps"], "views": {}}
    psi, phi = _view(state)
    shape = (s.n_cells, s.M)
    whole = psi if psi.shape == shape else torch.empty(shape, dtype=psi.dtype, device="cuda")
    _fill(whole, phi, case, seed, quad[3])
    if whole is not psi:
        psi.copy_(whole.view(psi.shape))
    return state


def run(state):
    if "batch" in state:
        b = state["batch"].step(state["steps"])
        q = [b.qoi(i) for i in range(state["members"])]
        keys = ("abs_now", "abs_int", "mass", "outflow_now", "outflow_int")
        return {k: torch.tensor(np.array([v[k] for v in q]), dtype=torch.float32) for k in keys}
    s = state["solver"].step(state["steps"])
    q = s.qoi()
    psi, phi = _view(state)
    return {"psi": psi, "phi": phi, "qoi": _now(q)}


def work(case):
    """A step reads the state once and writes it once; about 15 operations per cell and
    ordinate and stage at first order, 40 at second order, twice that with the
    limited gradients on triangles."""
    size = 2 if case["storage"] == "bf16" else 4
    if case["kind"] == "sweep":
        values = sum(n * n * M for n, M, _, _ in _members(case, 0))
    else:
        values = case["n"] ** 2 * case["M"] * (2 if case["kind"] == "enclosure" else 1)
    ops = 15 if case["order"] == 1 else 80 if case["kind"] == "enclosure" else 40
    return {"bytes": 2 * size * values * case["steps"], "flops": ops * values * case["steps"] * (2 if case["heun"] else 1)}


# ---------------------------------------------------------------------------- the same in 64 bits
def _minmod(a, b):
    return torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))


class _Grid:
    """The lattice: dpsi/dt = -div + ... with upwind or MUSCL-minmod faces, vacuum outside."""

    def __init__(self, p, quad, order):
        m = p.mesh
        self.n, self.h, self.order = m.nx, (m.dx, m.dy), order
        self.area = torch.full((m.n_cells,), m.dx * m.dy, dtype=torch.float64, device="cuda")
        self.boxes = [[int(round(v / m.dx)) for v in b] for b in p.extra.get("boxes", ())]

    def faces(self, P, v, d):
        """Upwind values on the n + 1 faces along axis d of P [ny, nx, ordinates]."""
        n = P.shape[d]
        ghost = torch.zeros_like(P.narrow(d, 0, 1))
        slope = 0.0
        if self.order == 2:
            slope = 0.5 * _minmod(torch.cat([P.narrow(d, 1, n - 1), ghost], d) - P, P - torch.cat([ghost, P.narrow(d, 0, n - 1)], d))
        up, down = P + slope, P - slope
        up.narrow(d, n - 1, 1).copy_(P.narrow(d, n - 1, 1))
        down.narrow(d, 0, 1).copy_(P.narrow(d, 0, 1))
        return torch.where(v > 0, torch.cat([ghost, up], d), torch.cat([down, ghost], d))

    def div(self, psi, xi, eta):
        P = psi.view(self.n, self.n, -1)
        out = 0.0
        for d, v in ((1, xi), (0, eta)):
            F = self.faces(P, v, d)
            out = out + v * (F.narrow(d, 1, self.n) - F.narrow(d, 0, self.n)) / self.h[1 - d]
        return out.view(psi.shape)

    def flows(self, psi, xi, eta, w):
        """Particle flow out of the domain and out of the boxes."""
        P = psi.view(self.n, self.n, -1)
        n, out = self.n, 0.0
        for cells, v, l in ((P[:, 0], -xi, 0), (P[:, n - 1], xi, 0), (P[0], -eta, 1), (P[n - 1], eta, 1)):
            out = out + self.h[1 - l] * (cells @ (w * v.clamp(min=0))).sum()
        boxes = []
        if self.boxes:
            X, Y = self.faces(P, xi, 1), self.faces(P, eta, 0)
            for i0, i1, j0, j1 in self.boxes:
                parts = ((X[j0:j1, i0], -xi, 0), (X[j0:j1, i1], xi, 0), (Y[j0, i0:i1], -eta, 1), (Y[j1, i0:i1], eta, 1))
                boxes.append(sum(self.h[1 - l] * (t @ (w * v.clamp(min=0))).sum() for t, v, l in parts))
        return out, boxes


class _Triangles:
    """The enclosure: upwind, or Green-Gauss gradients with the Venkatakrishnan limiter as the
    paper prints it; psi^- = 1 enters through x = 0. Cells in the solver's order."""

    def __init__(self, n, order):
        m = _mesh(n)
        perm = m["perm"]
        rank = np.empty_like(perm)
        rank[perm] = np.arange(perm.size)
        gpu = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
        self.order = order
        self.area, self.nl = gpu(m["area"][perm]), gpu(m["nl"][perm])
        nbr = m["nbr"][perm]
        self.inside = gpu(nbr >= 0)[:, :, None]
        self.nbr = gpu(np.where(nbr >= 0, rank[nbr], 0))
        self.inflow = gpu(m["side"][perm] == 0)[:, :, None]
        r = m["mid"] - m["cen"][:, None, :]
        self.r = gpu(r[perm])
        s = m["mid"] - np.where(m["nbr"][..., None] >= 0, m["cen"][m["nbr"]], 0.0)   # midpoint seen from the neighbour
        self.s = gpu(s[perm])

    def across(self, psi, e, xi):
        ghost = torch.where(self.inflow[:, e] & (xi > 0), 1.0, 0.0).to(psi.dtype)
        return torch.where(self.inside[:, e], psi[self.nbr[:, e]], ghost)

    def gradient(self, psi, xi):
        o = [self.across(psi, e, xi) for e in range(3)]
        gx = sum(self.nl[:, e, 0:1] * (0.5 * (psi + o[e])) for e in range(3)) / self.area[:, None]
        gy = sum(self.nl[:, e, 1:2] * (0.5 * (psi + o[e])) for e in range(3)) / self.area[:, None]
        top = torch.maximum(torch.maximum(o[0], o[1]), torch.maximum(o[2], psi)) - psi
        low = torch.minimum(torch.minimum(o[0], o[1]), torch.minimum(o[2], psi)) - psi
        e2 = (self.area[:, None] ** 3) ** 2
        L = None
        for e in range(3):
            D = 0.5 * (gx * self.r[:, e, 0:1] + gy * self.r[:, e, 1:2])
            b = torch.where(D > 0, top, low)
            f = ((b * b + e2) * D + 2 * D * D * b) / (b * b + 2 * D * D + b * D + e2) / D
            f = torch.where(D == 0, torch.ones_like(f), f)
            L = f if L is None else torch.minimum(L, f)
        return L * gx, L * gy

    def div(self, psi, xi, eta):
        if self.order == 2:
            gx, gy = self.gradient(psi, xi)
        out = 0.0
        for e in range(3):
            on = self.nl[:, e, 0:1] * xi + self.nl[:, e, 1:2] * eta
            mine, other = psi, self.across(psi, e, xi)
            if self.order == 2:
                j = self.nbr[:, e]
                mine = torch.where(self.inside[:, e], psi + gx * self.r[:, e, 0:1] + gy * self.r[:, e, 1:2], psi)
                other = torch.where(self.inside[:, e], other + gx[j] * self.s[:, e, 0:1] + gy[j] * self.s[:, e, 1:2], other)
            out = out + on * torch.where(on > 0, mine, other)
        return out / self.area[:, None]

    def flows(self, psi, xi, eta, w):
        out = 0.0
        for e in range(3):
            at = (~self.inside[:, e, 0]).nonzero()[:, 0]
            on = self.nl[at, e, 0:1] * xi + self.nl[at, e, 1:2] * eta
            ghost = torch.where(self.inflow[at, e] & (xi > 0), 1.0, 0.0).to(psi.dtype)
            out = out + ((on * torch.where(on > 0, psi[at], ghost)) @ w).sum()
        return out, []


def _solve(op, psi, p, quad, dt, heun, steps, order_of_cells):
    """`steps` steps from psi [cell][ordinate] in 64 bits, 64 ordinates at a time."""
    gpu = lambda a: torch.as_tensor(np.asarray(a, dtype=np.float64), device="cuda")  # noqa: E731
    xi, eta, w = gpu(quad[0]), gpu(quad[1]), gpu(quad[3])
    mats = np.asarray(p.materials.cell_mat)[order_of_cells]
    mt = p.materials
    sa, ss, q = gpu(mt.sigma_a[mats]), gpu(mt.sigma_s[mats]), gpu(mt.Q[mats])
    region = torch.as_tensor(np.asarray(mt.cell_region)[order_of_cells], device="cuda")
    blocks = [slice(k, k + 64) for k in range(0, psi.shape[1], 64)]

    def stage(u, base):
        phi = u @ w
        gain = (ss * phi / (2 * np.pi) + q)[:, None]
        out = torch.empty_like(u)
        for k in blocks:
            part = u[:, k].contiguous()
            v = part + dt * (gain - (sa + ss)[:, None] * part - op.div(part, xi[k], eta[k]))
            out[:, k] = v if base is None else 0.5 * (base[:, k] + v)
        return out

    def integrands(u):
        phi = u @ w
        a = op.area * sa * phi
        flows = [op.flows(u[:, k].contiguous(), xi[k], eta[k], w[k]) for k in blocks]
        return {"abs": [float(a[region == r].sum()) for r in range(mt.n_regions)], "mass": float((op.area * phi).sum()),
                "outflow": float(sum(f[0] for f in flows)), "box_out": [float(sum(v)) for v in zip(*(f[1] for f in flows))]}

    for _ in range(steps):
        one = stage(psi, None)
        psi = stage(one, psi) if heun else one
    return psi, psi @ w, integrands(psi)


def exact(case, seed):
    if case["kind"] == "sweep":
        rows = {k: [] for k in ("abs_now", "abs_int", "mass", "outflow_now", "outflow_int")}
        for n, M, sa, ss in _members(case, seed):
            p = _member_problem(n, sa, ss)
            psi = torch.zeros((n * n, M), dtype=torch.float64, device="cuda")
            _, _, S = _solve(_Grid(p, _quad(M), case["order"]), psi, p, _quad(M), 0.5 * p.mesh.dx, case["heun"],
                             BATCH_SPIN_UP + case["steps"], slice(None))
            rows["abs_now"].append(S["abs"])
            rows["mass"].append(S["mass"])
            rows["outflow_now"].append(S["outflow"])
        return {k: torch.tensor(v, dtype=torch.float64) if v else None for k, v in rows.items()}
    p, quad, dt = _setup(case, seed)
    lattice = case["kind"] == "lattice"
    op = _Grid(p, quad, case["order"]) if lattice else _Triangles(case["n"], case["order"])
    psi = torch.empty((p.mesh.n_cells, case["M"]), dtype=torch.bfloat16 if case["storage"] == "bf16" else torch.float32,
                      device="cuda")
    _fill(psi, None, case, seed, quad[3])
    psi, phi, S = _solve(op, psi.double(), p, quad, dt, case["heun"], case["steps"],
                            slice(None) if lattice else _mesh(case["n"])["perm"])
    if case["M"] not in PRODUCT and _regrouped(case["M"]):
        psi = psi.view(-1, 4, case["M"] // 4)
    return {"psi": psi, "phi": phi, "qoi": S}


def _regrouped(M):
    """Whether a Cartesian solver of M tessellation ordinates keeps its quadrants apart: each is then padded
    to a multiple of 64, for at most an eighth more ordinates."""
    per, Mpad = M // 4, -(-M // 32) * 32
    return any(per % c and 4 * (-(-per // c) * c) <= Mpad + Mpad // 8 for c in (128, 64))
