"""The update psi + dt F of the triangle kernels rounds F and the sum, nothing else."""
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


def fma(a, b, c):
    return (np.float64(a) * b.astype(np.float64) + c).astype(f32)


@pytest.mark.parametrize("order,staged", [(1, 1), (1, 0), (2, None)])
@pytest.mark.parametrize("heun", [False, True])
@pytest.mark.parametrize("n_p,n_phi", [(2, 16), (4, 16), (8, 16)])   # 1, 2 and 4 ordinates per lane
def test_decay_of_a_uniform_state(rt, order, staged, heun, n_p, n_phi):
    """A state that is uniform in space in a pure absorber: F = -sigma_t psi away from the sides, so that psi follows a
    recursion of a few roundings a stage. sigma_t and dt are floats whose product is none (its rounding would be off
    by the same amount in every step)."""
    sigma, dt, steps = float(f32(119.3)), 3 * 2.0 ** -11, 3 if heun else 6
    mesh = si.split_grid_mesh(24, 1.0, jitter=0.2, seed=4)
    n, M = mesh.n_cells, n_p * n_phi
    mats = si.Materials(sigma_a=np.array([sigma]), sigma_s=np.array([0.0]), Q=np.array([0.0]), cell_mat=np.zeros(n, np.int32),
                        cell_region=np.zeros(n, np.int32), region_names=("all",))
    p = si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=1024 * dt)
    s = rt.Solver(p, rt.rt_quad_product(n_p, n_phi), order=order, integrator=rt.RT_HEUN if heun else rt.RT_EULER, dt=dt)
    if staged is not None:
        rt.rt_debug_set(s.h, "tri_staged", staged)
    assert s.info.dt == dt
    c = np.linspace(0.5, 1.0, M).astype(f32)   # psi^n by ordinate
    s.set_psi(np.tile(c, (n, 1)))
    s.step(steps)
    psi = s.psi()
    s.close()
    centre = mesh.vertices[mesh.triangles].mean(axis=1)
    away = np.all(np.abs(centre - 0.5) < 0.15, axis=1)   # 8 cells of the grid from the sides, 6 stages
    for _ in range(steps):
        one = fma(f32(dt), -(f32(sigma) * c), c)
        if heun and order == 1:
            one = f32(0.5) * (c + fma(f32(dt), -(f32(sigma) * one), one))
        elif heun:
            one = f32(0.5) * fma(f32(dt), -(f32(sigma) * one), c + one)
        c = one
    assert away.sum() > 40 and np.array_equal(psi[away], np.tile(c, (away.sum(), 1)))


def second_order_euler(mesh, quad, psi, sigma, dt):
    """One Euler step of the limited scheme in a pure absorber with vacuum sides, operation by operation as the
    kernels compute it, with rounded quotients in the limiter."""
    V, T = mesh.vertices, mesh.triangles
    n, M = psi.shape
    P = V[T]
    Q = np.roll(P, -1, axis=1)
    A = 0.5 * ((P[:, 1, 0] - P[:, 0, 0]) * (P[:, 2, 1] - P[:, 0, 1]) - (P[:, 1, 1] - P[:, 0, 1]) * (P[:, 2, 0] - P[:, 0, 0]))
    cen = (P[:, 0] + P[:, 1] + P[:, 2]) / 3.0
    side = {}
    nbr = np.full((n, 3), -1)
    for t in range(n):
        for e in range(3):
            key = frozenset((T[t, e], T[t, (e + 1) % 3]))
            if key in side:
                u, f = side[key]
                nbr[t, e], nbr[u, f] = u, t
            else:
                side[key] = t, e
    inside = (nbr >= 0)[:, :, None]
    ax, ay = ((Q[..., 1] - P[..., 1]) / A[:, None]).astype(f32), (-(Q[..., 0] - P[..., 0]) / A[:, None]).astype(f32)
    r = (0.5 * (P + Q) - cen[:, None]).astype(f32)
    s = np.where(inside, 0.5 * (P + Q) - cen[nbr], 0.0).astype(f32)
    eps2 = ((A * A * A) ** 2).astype(f32)[:, None]
    c = psi
    nb = [np.where(inside[:, e], psi[nbr[:, e]], f32(0)) for e in range(3)]
    h = f32(0.5)
    d3 = [v - c for v in nb]

    def fm(a, b, x):
        return (np.float64(1) * a * b.astype(np.float64) + x).astype(f32)

    gx, gy = (fm(h * a[:, 2:3], d3[2], fm(h * a[:, 1:2], d3[1], h * a[:, 0:1] * d3[0])) for a in (ax, ay))
    up, dn = np.maximum(np.maximum.reduce(d3), 0), -np.minimum(np.minimum.reduce(d3), 0)
    def limiter(scale):
        """(smallest of the three edges' values, smallest denominator); x and y times 2^63 where den < 2^-100 if asked for."""
        L = lo = None
        for e in range(3):
            D = fm(h * r[:, e, 1:2], gy, h * r[:, e, 0:1] * gx)
            x, y = np.abs(D), np.where(D > 0, up, dn)
            den = fm(x + x, x, fm(y, y, eps2) + x * y)
            k = np.where(scale & (den < f32(2.0 ** -100)), f32(2.0 ** 63), f32(1))
            x, y = x * k, y * k
            p = x * y
            q = fm(y, y, eps2 * k * k) + p
            den = fm(x + x, x, q)
            one = (q + p) / den
            L, lo = (one, den) if L is None else (np.minimum(L, one), np.minimum(lo, den))
        return L, lo

    L, lo = limiter(False)
    if lo.min() < 2.0 ** -118:   # the kernels rescale where residuals would leave the range of floats
        pair = M > 32            # (both values of a lane's pair together)
        low = lo < f32(2.0 ** -118)
        low = (low | np.stack([low[:, 1::2], low[:, ::2]], 2).reshape(low.shape)) if pair else low
        L = np.where(low, limiter(True)[0], L)
    lx, ly = L * gx, L * gy
    div = np.zeros_like(c)
    xi, eta = (np.asarray(v, f32)[None] for v in quad[:2])
    for e in range(3):
        on = fm(eta, np.broadcast_to(ay[:, e:e + 1], c.shape), xi * ax[:, e:e + 1])
        mine = fm(lx, r[:, e, 0:1], ly * r[:, e, 1:2])
        other = fm(lx[nbr[:, e]], s[:, e, 0:1], fm(ly[nbr[:, e]], s[:, e, 1:2], d3[e]))
        mine = np.where(inside[:, e], mine, f32(0))
        other = np.where(inside[:, e], other, d3[e])
        div = fm(on, np.where(on > 0, mine, other), div)
    return fm(f32(dt), fm(np.full_like(c, -f32(sigma)), c, -div), c)


@pytest.mark.parametrize("n_p,n_phi", [(2, 16), (4, 16), (8, 16)])   # 1, 2 and 4 ordinates per lane
@pytest.mark.parametrize("L,scale", [(1.0, 1.0), (0.01, 1.0), (1.0, 1e-17), (0.01, 1e-18)])
def test_limiter_divides_to_the_last_bit(rt, n_p, n_phi, L, scale):
    """Every other cell is empty, so that a step leaves dt F there and the limiter's last bits show: equal but for
    values that the 64-bit stand-in of a fused operation rounds twice, or a quotient within 2^-21 ulp of the middle
    between two floats (1e-4 of the values: 36 quotients reach a value, with its neighbours')."""
    mesh = si.split_grid_mesh(21, L, jitter=0.2, seed=4)
    n, M, sigma = mesh.n_cells, n_p * n_phi, 3.0
    mats = si.Materials(sigma_a=np.array([sigma]), sigma_s=np.array([0.0]), Q=np.array([0.0]), cell_mat=np.zeros(n, np.int32),
                        cell_region=np.zeros(n, np.int32), region_names=("all",))
    quad = rt.rt_quad_product(n_p, n_phi)
    s = rt.Solver(si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=1.0), quad, order=2, integrator=rt.RT_EULER)
    psi0 = (si.random_psi(n, M, seed=6) * (np.arange(n) % 2)[:, None] * scale).astype(f32)
    s.set_psi(psi0)
    s.step(1)
    psi, dt = s.psi(), s.info.dt
    s.close()
    assert np.mean(psi != second_order_euler(mesh, quad, psi0, sigma, dt)) <= 1e-4


@pytest.mark.parametrize("vec", [0, 1])   # the streaming and the general kernel
@pytest.mark.parametrize("lane", [0, 13, 31])
def test_quantities_are_summed_in_64_bits(rt, vec, lane):
    """Scalar fluxes that any FP64 sum adds exactly (they span 53 bits) and an FP32 sum with one term for its errors
    does not, in the eight cells that one lane adds. One ordinate without a direction and with weight 1, so that
    phi = psi, unit cells of nothing, one cell per thread of a block."""
    n = 48
    mesh = si.CartesianMesh(nx=n, ny=n, x0=0.0, y0=0.0, dx=1.0, dy=1.0)
    mats = si.Materials(sigma_a=np.zeros(1), sigma_s=np.zeros(1), Q=np.zeros(1), cell_mat=np.zeros(n * n, np.int32),
                        cell_region=np.zeros(n * n, np.int32), region_names=("all",))
    p = si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=10.0)
    psi = np.zeros((n, n))
    for j, v in enumerate([2.0 ** 26, 1.0, 2.0 ** -25, 2.0 ** -25, -2.0 ** 26, -1.0, 2.0 ** -24, 0.0]):
        t = lane + 32 * j
        psi[16 + t // 16, 32 + t % 16] = v
    one = (np.zeros(1), np.zeros(1), np.ones(1), np.ones(1))
    s = rt.Solver(p, one, order=1, integrator=rt.RT_EULER, dt=1.0, tile_x=16, tile_y=16, vec=vec)
    s.set_psi(psi.reshape(-1, 1))
    s.step(2)
    q, got = s.qoi(), s.psi()
    s.close()
    assert np.array_equal(got[:, 0], psi.ravel())
    assert q["mass"] == 2.0 ** -23


def test_heun_average_rounds_once_at_the_size_of_psi(rt):
    """Above 1e5 cells the streaming kernel sums differences. Stage 2 adds the update in half its size and psi^n / 2 in
    one fused operation (psi^n + a psi first, and the differences to their half, rounds twice at the size of psi). All
    ordinates flow towards +x, +y; cells three or more from the sides, operation by operation."""
    nx, ny, sigma, q, dt = 420, 250, 3.0, 0.3, 2.0 ** -6
    xi, eta, mu, w = rt.rt_quad_product(16, 32)
    k = np.nonzero((xi > 0) & (eta > 0))[0][:32]
    quad = tuple(v[k] for v in (xi, eta, mu, w))
    mesh = si.CartesianMesh(nx=nx, ny=ny, x0=0.0, y0=0.0, dx=0.04, dy=0.05)
    mats = si.Materials(sigma_a=np.array([sigma]), sigma_s=np.zeros(1), Q=np.array([q]), cell_mat=np.zeros(nx * ny, np.int32),
                        cell_region=np.zeros(nx * ny, np.int32), region_names=("all",))
    s = rt.Solver(si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=64 * dt), quad, order=2,
                  integrator=rt.RT_HEUN, dt=dt)
    psi0 = (0.5 + si.random_psi(nx * ny, 32, seed=2)).astype(f32)
    s.set_psi(psi0)
    s.step(1)
    got = s.psi().reshape(ny, nx, 32)
    assert s.info.dt == dt
    s.close()
    h, one = f32(0.5), np.float64(1)

    def fm(a, b, x):
        return (one * a * b.astype(np.float64) + x).astype(f32)

    def minmod(a, b):
        return np.where(a * b > 0, np.where(np.abs(a) < np.abs(b), a, b), f32(0))

    a, b = fm(-f32(dt), np.full((1,), f32(sigma)), f32(1)), f32(dt) * f32(q)
    ax, ay = (f32(dt) * np.asarray(v, f32)[k] * f32(1.0 / d) for v, d in ((xi, mesh.dx), (eta, mesh.dy)))

    def stage(u, base):
        c = f32(1) if base is None else h
        dx, dy = np.diff(u, axis=1, prepend=f32(0)), np.diff(u, axis=0, prepend=f32(0))
        mx, my = minmod(dx[:, 1:], dx[:, :-1]), minmod(dy[1:], dy[:-1])          # of cells 0 .. n - 2
        mx, my = np.concatenate([mx, mx[:, :1]], 1), np.concatenate([my, my[:1]], 0)   # (the last cells are not looked at)
        g = fm(h, mx - np.roll(mx, 1, 1), dx)
        z = (-c * ax) * g
        low = h * np.roll(my, 1, 0)
        z = fm(np.broadcast_to(-c * ay, u.shape), dy - low, z)
        out = fm(np.broadcast_to(-c * ay, u.shape), h * my, z)
        t = fm(c * a, u, c * b) + out
        return t if base is None else fm(h, base, t)

    u = psi0.reshape(ny, nx, 32)
    want = stage(stage(u, None), u)
    inner = np.s_[6:-6, 6:-6]
    assert np.mean(got[inner] != want[inner]) <= 1e-5   # (fused operations that the 64-bit stand-in rounds twice)
