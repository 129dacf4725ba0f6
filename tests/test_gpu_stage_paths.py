"""Edges of the stage kernels' dispatch and reductions, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import sn_inputs as si

pytestmark = pytest.mark.gpu

PSI_TOL = 1e-5      # FP32 storage, relative L2 of psi
QOI_TOL = 1e-4


@pytest.fixture(scope="module")
def rt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2505_17284_gb300 import build, rt as rtmod
    build.build()
    rtmod.load_library()
    return rtmod


def rel_l2(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


@pytest.mark.parametrize("kind,M", [("cart", (2, 16)), ("cart", (8, 16)), ("tri", (2, 16))])
@pytest.mark.parametrize("regions", [1, 7, 16])
def test_qoi_sums_of_many_regions(rt, kind, M, regions):
    """Up to 16 QoI regions, scattered over the cells (with the smallest ring of the
    Cartesian kernels they are summed in several rounds): absorption per region,
    mass and outflow of the current state and their time integrals."""
    p = si.lattice_problem(35) if kind == "cart" else si.lattice_triangle_problem(12, jitter=0.2, seed=3)
    m = p.materials
    m.cell_region = (np.arange(p.mesh.n_cells) * 7 % regions).astype(np.int32)
    m.region_names = tuple(f"r{i}" for i in range(regions))
    m.sigma_a = np.array([0.3, 10.0, 0.7])
    psi0 = si.random_psi(p.mesh.n_cells, M[0] * M[1], seed=regions)
    s = rt.Solver(p, rt.rt_quad_product(*M))
    s.set_psi(psi0)
    s.step(3)
    psi, q, dt = s.psi(), s.qoi(), s.info.dt
    s.close()
    op = (oracle.CartesianOracle if kind == "cart" else oracle.TriangleOracle)(p, oracle.product_quadrature(*M), order=1)
    ref, acc, S = oracle.run(op, psi0, dt, 3, "euler")
    assert rel_l2(psi, ref) <= PSI_TOL
    assert np.allclose(q["abs_now"], S["abs"], rtol=QOI_TOL, atol=1e-3 * QOI_TOL * S["mass"])
    assert np.allclose(q["abs_int"], acc.abs_int, rtol=QOI_TOL, atol=1e-3 * QOI_TOL * S["mass"])
    assert abs(q["mass"] - S["mass"]) <= QOI_TOL * S["mass"]
    assert abs(q["outflow_now"] - S["outflow"]) <= QOI_TOL * max(abs(S["outflow"]), 1e-3 * S["mass"])
    assert abs(q["outflow_int"] - acc.outflow_int) <= QOI_TOL * max(abs(acc.outflow_int), 1e-3 * S["mass"])


def cart_problem(nx, ny, seed, periodic=(False, False)):
    """Random materials and regions on an nx x ny grid, inflow on every side (or periodic axes)."""
    rng = np.random.default_rng(seed)
    mesh = si.CartesianMesh(nx=nx, ny=ny, x0=0.0, y0=0.0, dx=0.1, dy=0.07)
    mats = si.Materials(sigma_a=rng.uniform(0, 5, 4), sigma_s=rng.uniform(0, 3, 4), Q=rng.uniform(0, 1, 4),
                        cell_mat=rng.integers(0, 4, nx * ny).astype(np.int32),
                        cell_region=rng.integers(0, 3, nx * ny).astype(np.int32), region_names=("a", "b", "c"))
    kind, inflow = [si.INFLOW] * 4, rng.uniform(0.2, 1.5, 4)
    for axis in range(2):
        if periodic[axis]:
            kind[2 * axis] = kind[2 * axis + 1] = si.PERIODIC
            inflow[2 * axis:2 * axis + 2] = 0.0
    return si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(tuple(kind), tuple(inflow)), t_end=1.0)


def quadratures(rt, name):
    """Quadratures by how their directions change along the ordinates."""
    kind, a = name.split("-")
    if kind == "prod":
        return rt.rt_quad_product(*[int(v) for v in a.split("x")])
    if kind == "tess":
        return rt.rt_quad_tessellation(int(a))
    xi, eta, mu, w = rt.rt_quad_product(4, 16)
    if kind == "axes":      # components that are exactly 0, at the runs' ends and inside them
        xi, eta = xi.copy(), eta.copy()
        xi[[0, 15, 20, 33]] = 0.0
        eta[[3, 31, 32, 40]] = 0.0
        xi[50], eta[50] = 0.0, 0.0
    if kind == "shuffled":  # signs change from ordinate to ordinate
        k = np.random.default_rng(int(a)).permutation(64)
        xi, eta, mu, w = xi[k], eta[k], mu[k], w[k]
    if kind == "first":     # a few ordinates only
        xi, eta, mu, w = (v[:int(a)] for v in (xi, eta, mu, w))
    return xi, eta, mu, w


@pytest.mark.parametrize("quad", ["prod-4x16", "prod-8x16", "prod-2x16", "prod-3x12", "prod-8x32", "tess-3", "tess-5",
                                  "tess-7", "tess-9", "axes-0", "shuffled-1", "first-1", "first-33"])
@pytest.mark.parametrize("order,heun", [(1, False), (2, True), (1, True), (2, False)])
def test_cartesian_stage_over_quadratures_and_ragged_tiles(rt, quad, order, heun):
    """Every way the ordinates fall into windows (whole, partial, mixed signs of xi, or
    none: the general kernel), on grids smaller than a tile, ragged in x and y, with
    segments from one row up, inflow on all sides."""
    q = quadratures(rt, quad)
    for i, (nx, ny, ty) in enumerate([(1, 1, 0), (3, 2, 1), (9, 7, 2), (17, 11, 3), (37, 21, 0), (40, 33, 16)]):
        p = cart_problem(nx, ny, seed=17 * i + order)
        psi0 = si.random_psi(p.mesh.n_cells, len(q[0]), seed=i)
        s = rt.Solver(p, q, order=order, integrator=rt.RT_HEUN if heun else rt.RT_EULER, dt=0.02, tile_y=ty)
        s.set_psi(psi0)
        s.step(3)
        psi, qoi, dt = s.psi(), s.qoi(), s.info.dt
        s.close()
        op = oracle.CartesianOracle(p, q, order=order)
        ref, acc, S = oracle.run(op, psi0, dt, 3, "heun" if heun else "euler")
        assert rel_l2(psi, ref) <= PSI_TOL, (nx, ny)
        assert abs(qoi["mass"] - S["mass"]) <= QOI_TOL * S["mass"], (nx, ny)
        assert abs(qoi["outflow_int"] - acc.outflow_int) <= QOI_TOL * max(abs(acc.outflow_int), 1e-3 * S["mass"]), (nx, ny)


@pytest.mark.parametrize("periodic", [(True, False), (False, True), (True, True)])
@pytest.mark.parametrize("quad", ["prod-4x16", "tess-5"])
def test_cartesian_stage_partial_windows_on_periodic_sides(rt, quad, periodic):
    q = quadratures(rt, quad)
    for nx, ny, ty in ((5, 4, 1), (18, 13, 4)):
        p = cart_problem(nx, ny, seed=5, periodic=periodic)
        psi0 = si.random_psi(p.mesh.n_cells, len(q[0]), seed=2)
        s = rt.Solver(p, q, order=2, integrator=rt.RT_HEUN, dt=0.02, tile_y=ty)
        s.set_psi(psi0)
        s.step(3)
        psi, dt = s.psi(), s.info.dt
        s.close()
        ref, _, _ = oracle.run(oracle.CartesianOracle(p, q, order=2), psi0, dt, 3, "heun")
        assert rel_l2(psi, ref) <= PSI_TOL, (nx, ny)


@pytest.mark.parametrize("quad", ["prod-4x16", "prod-8x16", "tess-5"])
def test_cartesian_stage_bf16_agrees_with_the_general_kernel(rt, quad):
    """BF16 storage: the streaming kernel and the general one (an explicit number of
    ordinates per lane) round with the same bits per (cell, ordinate, step, stage), so
    after one Euler step nearly all stored values agree exactly, and both are within
    BF16's unit roundoff (2^-8, stochastic rounding) of the oracle."""
    q = quadratures(rt, quad)
    p = cart_problem(37, 21, seed=3)
    psi0 = si.random_psi(p.mesh.n_cells, len(q[0]), seed=4)
    out = []
    for vec in (0, 1):
        s = rt.Solver(p, q, order=2, integrator=rt.RT_EULER, storage=rt.RT_BF16, dt=0.02, vec=vec)
        s.set_psi(psi0)
        start, dt = s.psi(), s.info.dt
        s.step(1)
        out.append(s.psi())
        s.close()
    ref, _, _ = oracle.run(oracle.CartesianOracle(p, q, order=2), start, dt, 1, "euler")
    assert np.mean(out[0] == out[1]) >= 0.995
    assert rel_l2(out[0], ref) <= 2.0 ** -8 and rel_l2(out[1], ref) <= 2.0 ** -8


def test_dropped_load_of_the_streaming_kernel_is_reported(rt):
    p = si.lattice_problem(35)
    s = rt.Solver(p, rt.rt_quad_product(4, 16), order=2, integrator=rt.RT_HEUN, dt=0.1)
    rt.rt_debug_set(s.h, "drop_load", 1)
    s.step(1)
    with pytest.raises(rt.RTError) as e:
        s.qoi()
    assert e.value.code == rt.RT_ETIMEOUT
    s.close()


@pytest.mark.parametrize("M", [(2, 16), (4, 16), (6, 16), (8, 16)])   # 1, 2, 1 and 4 ordinates per lane
@pytest.mark.parametrize("scale", [1e-16, 1e-9, 1.0, 1e18])
def test_second_order_triangles_over_scales_of_the_state(rt, M, scale):
    """The limiter divides with a fast quotient inside its range and by IEEE division
    outside it (states below 1e-15 or above 1e18): the scheme is homogeneous in the
    state and source, so every scale must match the oracle alike."""
    mesh = si.split_grid_mesh(13, 0.01, jitter=0.2, seed=4)   # cells so small that epsilon^2 is far below beta^2
    n = mesh.n_cells
    mats = si.Materials(sigma_a=np.array([1.0, 40.0]), sigma_s=np.array([20.0, 3.0]), Q=np.array([0.5, 30.0]) * scale,
                        cell_mat=(np.arange(n) // 5 % 2).astype(np.int32), cell_region=np.zeros(n, np.int32),
                        region_names=("all",))
    p = si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=1.0)
    psi0 = (si.smooth_psi(mesh, M[0] * M[1], seed=2) + 0.2 * si.random_psi(n, M[0] * M[1], seed=3)) * scale
    s = rt.Solver(p, rt.rt_quad_product(*M), order=2, integrator=rt.RT_HEUN)
    s.set_psi(psi0)
    s.step(2)
    psi, dt = s.psi(), s.info.dt
    s.close()
    op = oracle.TriangleOracle(p, oracle.product_quadrature(*M), order=2)
    ref, _, _ = oracle.run(op, psi0, dt, 2, "heun")
    assert rel_l2(psi, ref) <= PSI_TOL


@pytest.mark.parametrize("integrator", ["euler", "heun"])
def test_first_order_triangle_quantities_over_many_chunks_per_block(rt, integrator):
    """11,025 chunks of 32 cells, about 36 per resident block: the FP32 sums of 32
    chunks that each warp records before it adds them in FP64, against the sums of the
    state itself in FP64. A recorded float has at most 32 additions of non-negative
    terms and each term 32 ordinates' worth: 64 * 2^-24 = 3.8e-6 at most."""
    p = si.enclosure_problem(420, jitter=0.2, seed=9)
    quad = rt.rt_quad_product(2, 16)
    op = oracle.TriangleOracle(p, oracle.product_quadrature(2, 16), order=1)
    w, area, sa = oracle.product_quadrature(2, 16)[3], op.area, p.materials.sigma_a[p.materials.cell_mat]
    psi0 = si.random_psi(p.mesh.n_cells, 32, seed=12)
    got = []
    for staged in (1, 0):
        s = rt.Solver(p, quad, order=1, integrator=rt.RT_HEUN if integrator == "heun" else rt.RT_EULER)
        rt.rt_debug_set(s.h, "tri_staged", staged)
        s.set_psi(psi0)
        s.step(2)
        phi = s.psi().astype(np.float64) @ w
        q = s.qoi()
        s.close()
        assert abs(q["mass"] - np.sum(area * phi)) <= 4e-6 * q["mass"]
        per = np.bincount(p.materials.cell_region, weights=area * sa * phi, minlength=p.materials.n_regions)
        assert np.max(np.abs(np.asarray(q["abs_now"]) - per)) <= 4e-6 * np.max(per)
        got.append(q)
    for k in ("mass", "abs_int", "outflow_int"):
        a, b = (np.asarray(g[k], float) for g in got)
        assert np.max(np.abs(a - b)) <= 8e-6 * np.max(np.abs(b)), k


@pytest.mark.parametrize("M", [(2, 16), (4, 16), (8, 16)])   # 1, 2 and 4 ordinates per lane
@pytest.mark.parametrize("scale", [0.0, 1e-18, 1e-19, 1e-20, 1e-25])
def test_second_order_triangles_with_denominators_below_the_fast_range(rt, M, scale):
    """States whose squared differences lie around epsilon^2 = A^6 (about 1e-39 here, below
    the normal range) and a state of zeros: the limiter rescales its quotients there.
    epsilon^2 itself is held to 2e-6 of its value, the limiter with it."""
    mesh = si.split_grid_mesh(13, 0.01, jitter=0.2, seed=4)
    n = mesh.n_cells
    mats = si.Materials(sigma_a=np.array([1.0, 40.0]), sigma_s=np.array([20.0, 3.0]),
                        Q=np.array([0.0, 30.0]) * (scale or 1.0), cell_mat=(np.arange(n) == 60).astype(np.int32),
                        cell_region=np.zeros(n, np.int32), region_names=("all",))
    p = si.Problem(mesh=mesh, materials=mats, boundary=si.Boundary(), t_end=1.0)
    psi0 = (si.smooth_psi(mesh, M[0] * M[1], seed=2) + 0.2 * si.random_psi(n, M[0] * M[1], seed=3)) * scale
    s = rt.Solver(p, rt.rt_quad_product(*M), order=2, integrator=rt.RT_HEUN)
    s.set_psi(psi0)
    s.step(3)
    psi, dt = s.psi(), s.info.dt
    s.close()
    op = oracle.TriangleOracle(p, oracle.product_quadrature(*M), order=2)
    ref, _, _ = oracle.run(op, psi0, dt, 3, "heun")
    assert rel_l2(psi, ref) <= PSI_TOL


@pytest.mark.parametrize("order,tile_x", [(2, 16), (1, 32)])
def test_tiles_of_256_ordinates_above_2_17_cells(rt, order, tile_x):
    """371^2 cells, quadrants of 64 ordinates: second order takes 16-cell tiles, first
    order 32-cell ones, and either agrees with the other width to FP32 rounding of a few
    steps (each value's operations are the same; only phi's order of summation differs)."""
    p = si.lattice_problem(371)
    quad = rt.rt_quad_product(8, 32)
    out = []
    for tx in (0, 32 if tile_x == 16 else 16):
        s = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN, dt=0.5 * p.mesh.dx, tile_x=tx)
        assert s.info.tile_x == (tx or tile_x)
        s.step(3)
        out.append(s.phi())
        s.close()
    assert np.max(np.abs(out[0] - out[1])) <= 1e-6 * np.max(np.abs(out[1]))
