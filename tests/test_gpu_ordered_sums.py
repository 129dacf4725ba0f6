"""Second order on small Cartesian grids keeps one order of operations: the limited scheme
at the default time step amplifies rounding from step to step, so a kernel that adds in
another order gives other values after a few dozen steps (1e-3 after 96)."""
import numpy as np
import pytest

import sn_inputs as si

pytestmark = pytest.mark.gpu
f32 = np.float32


@pytest.fixture(scope="module")
def rt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2505_17284_gb300 import build, rt as rtmod
    build.build()
    rtmod.load_library()
    return rtmod


def problem(nx, ny, seed, periodic=False):
    """The lattice's cross-sections scattered over the cells, inflow on every side (or periodic axes)."""
    rng = np.random.default_rng(seed)
    mesh = si.CartesianMesh(nx=nx, ny=ny, x0=0.0, y0=0.0, dx=0.05, dy=0.05)
    mats = si.Materials(sigma_a=np.array([0.0, 12.0, 0.0]), sigma_s=np.array([1.2, 0.0, 0.7]), Q=np.array([0.0, 0.0, 1.0]),
                        cell_mat=rng.integers(0, 3, nx * ny).astype(np.int32),
                        cell_region=np.zeros(nx * ny, np.int32), region_names=("all",))
    bc = si.Boundary((si.PERIODIC,) * 4, (0.0,) * 4) if periodic else si.Boundary((si.INFLOW,) * 4, (0.3, 0.0, 1.1, 0.2))
    return si.Problem(mesh=mesh, materials=mats, boundary=bc, t_end=100.0)


def state(p, M, seed):
    return si.smooth_psi(p.mesh, M, seed=seed) * (1 + 0.1 * si.random_psi(p.mesh.n_cells, M, seed=seed + 1))


def after(rt, p, quad, psi0, steps, **options):
    s = rt.Solver(p, quad, order=2, dt=0.025, **options)
    s.set_psi(psi0)
    s.step(steps)
    got = s.psi(), s.phi(), s.info
    s.close()
    return got


@pytest.mark.parametrize("n_p,n_phi,vec", [(4, 16, 2), (6, 32, 2), (8, 16, 4), (8, 32, 4), (16, 32, 4)])
@pytest.mark.parametrize("nx,ny,tile_y,periodic", [(70, 70, 0, False), (93, 41, 0, False), (200, 64, 0, False), (31, 57, 2, True),
                                                   (9, 3, 7, False), (61, 70, 63, False)])
def test_streaming_and_general_kernel_store_the_same_bits(rt, n_p, n_phi, vec, nx, ny, tile_y, periodic):
    """psi and phi after 96 Heun steps from the kernel that the library picks (the streaming one, or the general
    one where so long a segment does not fit) and from the general one (an explicit number of ordinates per lane)."""
    p, quad = problem(nx, ny, seed=nx, periodic=periodic), rt.rt_quad_product(n_p, n_phi)
    psi0 = state(p, n_p * n_phi, seed=ny)
    a = after(rt, p, quad, psi0, 96, integrator=rt.RT_HEUN, variant=1, tile_y=tile_y)
    b = after(rt, p, quad, psi0, 96, integrator=rt.RT_HEUN, variant=1, vec=vec, tile_y=16)
    assert a[2].vec == 0 or tile_y == 63
    assert b[2].vec == vec
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("quad,vec", [("tess-3", 1), ("tess-5", 0), ("tess-7", 0), ("tess-9", 0), ("prod-6x16", 0)])
@pytest.mark.parametrize("nx,ny,tile_y,periodic", [(70, 70, 0, False), (93, 41, 0, False), (31, 57, 2, True), (9, 3, 7, False),
                                                   (61, 70, 63, False)])
def test_rules_of_one_ordinate_per_lane(rt, quad, vec, nx, ny, tile_y, periodic):
    """The same where quadrants are no multiples of two ordinates, so that windows are partial (tess-3 allows none)."""
    p = problem(nx, ny, seed=2, periodic=periodic)
    q = rt.rt_quad_tessellation(int(quad[5:])) if quad[0] == "t" else rt.rt_quad_product(*map(int, quad[5:].split("x")))
    psi0 = state(p, len(q[0]), seed=5)
    a = after(rt, p, q, psi0, 96, integrator=rt.RT_HEUN, variant=1, tile_y=tile_y)
    b = after(rt, p, q, psi0, 96, integrator=rt.RT_HEUN, variant=1, vec=1, tile_y=16)
    assert a[2].vec in (vec, 1)   # (1 where so long a segment does not fit)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


@pytest.mark.parametrize("n_p,n_phi,tile_y,integrator", [(9, 32, 8, "HEUN"), (11, 32, 8, "EULER"), (9, 32, 0, "HEUN")])
def test_segments_at_the_limit_of_shared_memory(rt, n_p, n_phi, tile_y, integrator):
    """8 rows of 288 ordinates (Heun; 352 in BF16 Euler) leave 112 bytes of a block's 227 KB: less than the kernel's own
    variables, so the general kernel takes them."""
    p, quad = problem(100, 64, seed=1), rt.rt_quad_product(n_p, n_phi)
    psi0 = state(p, n_p * n_phi, seed=4)
    storage = rt.RT_BF16 if integrator == "EULER" else rt.RT_FP32
    options = dict(integrator=getattr(rt, "RT_" + integrator), variant=1, storage=storage)
    a = after(rt, p, quad, psi0, 3, tile_y=tile_y, **options)
    b = after(rt, p, quad, psi0, 3, tile_y=8, vec=1, **options)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def fma(a, b, c):
    """a b + c in one rounding (the product of two floats is exact in 64 bits)."""
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(f32)


def stage(p, quad, psi, phi, dt, V, uniform):
    """One Euler stage of the second-order scheme, value by value as a lane computes it, and its phi: lanes of V
    ordinates, chunks of 32 V. Vacuum and inflow sides."""
    m, mt = p.mesh, p.materials
    xi, eta, w = (np.asarray(quad[i], f32) for i in (0, 1, 3))
    mats = np.asarray(mt.cell_mat).reshape(m.ny, m.nx)
    sa, ss, q = (np.asarray(v)[mats] for v in (mt.sigma_a, mt.sigma_s, mt.Q))
    dt = f32(dt)
    a = fma(np.full(mats.shape, -dt), (sa + ss).astype(f32), np.ones(mats.shape, f32))
    b = dt * fma((ss / (2 * np.pi)).astype(f32), phi.reshape(mats.shape).astype(f32), q.astype(f32))
    out = np.empty((m.ny, m.nx, len(xi)), f32)
    half = f32(0.5)

    def minmod(x, y):
        return np.where(x * y > 0, np.where(np.abs(x) < np.abs(y), x, y), f32(0))

    def faces(u, axis, sign, ghost, down):
        """Differences of the face values along the flow."""
        u = np.moveaxis(u, axis, 0)[::sign]
        n = u.shape[0]
        up = np.concatenate([np.full_like(u[:1], ghost), u])           # upwind cells of faces 0 .. n
        dn = np.concatenate([u, np.zeros_like(u[:1])])
        M = np.zeros_like(up)
        M[1:n] = minmod(u[1:] - u[:-1], up[1:n] - up[:n - 1])          # domain faces are first order
        if down:                                                        # the general kernel walks +y whatever the flow
            up = dn + (up - dn)
        F = fma(np.full_like(M, half), M, up)
        return np.moveaxis((F[1:] - F[:-1])[::sign], 0, axis)

    ghost = [f32(v) for v in p.boundary.inflow]
    inv = f32(1.0 / m.dx), f32(1.0 / m.dy)
    for k in range(len(xi)):
        u = psi[:, k].reshape(m.ny, m.nx).astype(f32)
        sx, sy = (1 if xi[k] > 0 else -1), (1 if eta[k] > 0 else -1)
        fx = faces(u, 1, sx, ghost[0 if sx > 0 else 1], False)
        fy = faces(u, 0, sy, ghost[2 if sy > 0 else 3], not uniform and sy < 0)
        ax, ay = (np.full_like(u, dt * abs(v) * i) for v, i in ((xi[k], inv[0]), (eta[k], inv[1])))
        div = fma(ax, fx, ay * fy) if uniform else fma(ay, fy, ax * fx)
        out[..., k] = fma(a, u, b) - div
    total = np.zeros(mats.shape, f32)
    for c in range(0, len(xi), 32 * V):
        lanes = []
        for k in range(c, c + 32 * V, V):
            t = [w[k + v] * out[..., k + v] for v in range(V)]
            if uniform:
                s = t[0] + t[1] if V == 2 else (fma(np.full_like(t[0], w[k + 2]), out[..., k + 2], t[0]) +
                                                fma(np.full_like(t[0], w[k + 3]), out[..., k + 3], t[1]))
            else:
                s = t[0]
                for v in range(1, V):
                    s = fma(np.full_like(s, w[k + v]), out[..., k + v], s)
            lanes.append(s)
        while len(lanes) > 1:
            h = len(lanes) // 2
            lanes = [x + y for x, y in zip(lanes[:h], lanes[h:])]
        total = total + lanes[0]
    return out.reshape(-1, len(xi)), total.ravel()


@pytest.mark.parametrize("n_p,n_phi,variant,tile_x,V", [(4, 16, 1, 0, 2), (8, 16, 1, 0, 4), (8, 32, 1, 16, 4), (8, 32, 2, 16, 2),
                                                        (8, 32, 2, 32, 2), (16, 32, 2, 0, 4), (16, 32, 1, 16, 4)])
def test_order_of_operations_of_a_stage(rt, n_p, n_phi, variant, tile_x, V):
    """Two Euler steps (the second one's source comes from the first one's phi) against the same operations in
    numpy, bit for bit but for values that the 64-bit stand-in of a fused operation rounds twice (1e-6 of them)."""
    p, quad = problem(37, 21, seed=8), rt.rt_quad_product(n_p, n_phi)
    psi0 = state(p, n_p * n_phi, seed=3).astype(f32)
    phi0 = after(rt, p, quad, psi0, 0, integrator=rt.RT_EULER, variant=variant, tile_x=tile_x)[1]
    got = after(rt, p, quad, psi0, 2, integrator=rt.RT_EULER, variant=variant, tile_x=tile_x)
    assert got[2].variant == variant
    psi, phi = stage(p, quad, psi0, phi0, got[2].dt, V, variant == 2)
    psi, phi = stage(p, quad, psi, phi, got[2].dt, V, variant == 2)
    assert np.mean(got[0] != psi) <= 1e-6 and np.mean(got[1] != phi) <= 1e-6


def test_batch_members_keep_their_bits(rt):
    """Members of every form in one batch: ordered with two blocks and with one block per SM (272^2 x 64), with one,
    two and four ordinates per lane, plain (330^2) and general (tess-3): psi and QoIs as alone, bit for bit."""
    members = [(272, "4x16"), (70, "4x16"), (96, "8x16"), (64, "16x32"), (50, "t5"), (330, "4x16"), (40, "t3"), (70, "4x16")]
    probs, quads = [], []
    for n, rule in members:
        p = si.lattice_problem(n)
        p.t_end = 100.0
        probs.append(p)
        quads.append(rt.rt_quad_tessellation(int(rule[1:])) if rule[0] == "t" else rt.rt_quad_product(*map(int, rule.split("x"))))
    b = rt.Batch(probs, quads, order=2, integrator=rt.RT_HEUN, dts=[0.5 * p.mesh.dx for p in probs])
    b.step(3)
    b.step(8)
    for i, (p, q) in enumerate(zip(probs, quads)):
        s = rt.Solver(p, q, order=2, integrator=rt.RT_HEUN, dt=0.5 * p.mesh.dx)
        s.step(11)
        mine, alone = b.qoi(i), s.qoi()
        for k in ("abs_now", "abs_int", "mass", "outflow_now", "outflow_int", "box_out_now"):
            assert np.array_equal(np.asarray(mine[k]), np.asarray(alone[k])), (members[i], k)
        assert np.array_equal(b.psi(i), s.psi()), members[i]
        s.close()
    b.close()
