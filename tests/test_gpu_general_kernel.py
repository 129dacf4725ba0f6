"""The general Cartesian kernel (an explicit number of ordinates per lane): its bounded waits, and its three widths at
the domain's sides against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import sn_inputs as si

pytestmark = pytest.mark.gpu

PSI_TOL = 1e-5      # FP32 storage, relative L2 of psi


@pytest.fixture(scope="module")
def rt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2505_17284_gb300 import build, rt as rtmod
    build.build()
    rtmod.load_library()
    return rtmod


@pytest.mark.parametrize("vec", [1, 2, 4])
@pytest.mark.parametrize("order,heun", [(1, False), (2, True)])
@pytest.mark.parametrize("load", [0, 3, 9])   # of the 10 rows or more that a segment of 8 pulls
def test_wait_for_a_dropped_load_runs_out(rt, vec, order, heun, load):
    """A row that never arrives: the wait for it gives up after the limit, the loads in flight are drained, the launch
    reports RT_ETIMEOUT, and the GPU stays usable. (The streaming kernel waits on no barrier that a load completes, so
    the wait is the general kernel's.)"""
    p, quad = si.lattice_problem(35), rt.rt_quad_product(8, 16)
    options = dict(order=order, integrator=rt.RT_HEUN if heun else rt.RT_EULER, dt=0.1, variant=1, vec=vec, tile_y=8)
    s = rt.Solver(p, quad, **options)
    assert s.info.variant == 1 and s.info.vec == vec
    rt.rt_debug_set(s.h, "wait_limit_cycles", 2_000_000)
    rt.rt_debug_set(s.h, "drop_load", load)
    s.step(1)
    with pytest.raises(rt.RTError) as e:
        s.qoi()
    assert e.value.code == rt.RT_ETIMEOUT and f"load {load}" in rt.rt_last_error()   # the wait that ran out
    with pytest.raises(rt.RTError) as e:
        s.step(1)
    assert e.value.code == rt.RT_ESTATE
    s.close()
    t = rt.Solver(p, quad, **options)
    t.step(3)
    assert t.qoi()["step"] == 3
    t.close()


@pytest.mark.parametrize("vec", [1, 2, 4])
@pytest.mark.parametrize("order,heun", [(1, False), (1, True), (2, False), (2, True)])
@pytest.mark.parametrize("periodic", [False, True])
def test_ordinates_per_lane_at_the_sides(rt, vec, order, heun, periodic):
    """Grids smaller than a tile and ragged in both axes, inflow on all sides or periodic axes."""
    quad = rt.rt_quad_product(8, 16)
    for i, (nx, ny, ty) in enumerate([(1, 1, 0), (9, 7, 2), (37, 21, 0), (40, 33, 16)]):
        rng = np.random.default_rng(i)
        mesh = si.CartesianMesh(nx=nx, ny=ny, x0=0.0, y0=0.0, dx=0.1, dy=0.07)
        mats = si.Materials(sigma_a=rng.uniform(0, 5, 4), sigma_s=rng.uniform(0, 3, 4), Q=rng.uniform(0, 1, 4),
                            cell_mat=rng.integers(0, 4, nx * ny).astype(np.int32),
                            cell_region=np.zeros(nx * ny, np.int32), region_names=("all",))
        bc = si.Boundary((si.PERIODIC,) * 4, (0.0,) * 4) if periodic else si.Boundary((si.INFLOW,) * 4, (0.4, 1.2, 0.7, 0.2))
        p = si.Problem(mesh=mesh, materials=mats, boundary=bc, t_end=1.0)
        psi0 = si.random_psi(nx * ny, 128, seed=i)
        s = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN if heun else rt.RT_EULER, dt=0.02, tile_y=ty, variant=1, vec=vec)
        assert s.info.variant == 1 and s.info.vec == vec
        s.set_psi(psi0)
        s.step(3)
        psi, dt = s.psi(), s.info.dt
        s.close()
        ref, _, _ = oracle.run(oracle.CartesianOracle(p, quad, order=order), psi0, dt, 3, "heun" if heun else "euler")
        assert np.linalg.norm(psi - ref) <= PSI_TOL * np.linalg.norm(ref), (nx, ny)
