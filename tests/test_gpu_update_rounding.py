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
