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
