"""The kernel options that the library reports and the tuner returns can be asked for, and the
tuner times the library's own choice and nothing twice."""
import numpy as np
import pytest

import sn_inputs as si

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rt():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2505_17284_gb300 import build, rt as rtmod
    build.build()
    rtmod.load_library()
    return rtmod


def options(s):
    return s.info.tile_x, s.info.tile_y, s.info.variant, s.info.vec


@pytest.mark.parametrize("rule", ["4x16", "8x16", "8x32", "16x32", "2x16", "tess-5", "tess-11", "one-quadrant"])
@pytest.mark.parametrize("n", [14, 70, 100, 280, 330, 380])
@pytest.mark.parametrize("order", [1, 2])
def test_reported_options_can_be_asked_for(rt, rule, n, order):
    if rule == "one-quadrant":
        xi, eta, mu, w = rt.rt_quad_product(16, 32)
        k = np.nonzero((xi > 0) & (eta > 0))[0][:64]
        quad = tuple(v[k] for v in (xi, eta, mu, w))
    else:
        quad = rt.rt_quad_tessellation(int(rule[5:])) if rule[0] == "t" else rt.rt_quad_product(*map(int, rule.split("x")))
    p = si.lattice_problem(n)
    a = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN)
    tx, ty, variant, vec = options(a)
    a.step(2)
    phi = a.phi()
    a.close()
    b = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN, tile_x=tx, tile_y=ty, variant=variant, vec=vec)
    assert options(b) == (tx, ty, variant, vec)
    b.step(2)
    assert np.array_equal(b.phi(), phi)
    b.close()


@pytest.mark.parametrize("rule,n,order,most", [((4, 16), 140, 2, 24), ((4, 16), 280, 1, 24), ((16, 32), 330, 2, 24),
                                               ((16, 32), 100, 1, 24), ((8, 16), 350, 2, 12)])
def test_tuner_builds_each_configuration_once(rt, monkeypatch, rule, n, order, most):
    """At most 12 segment lengths (one of them automatic) for each tile width, the library's own width among them."""
    import torch
    p, quad = si.lattice_problem(n), rt.rt_quad_product(*rule)
    own = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN)
    psi_bytes, width = int(own.info.n_cells) * int(own.info.M_pad) * 4, own.info.tile_x
    own.close()
    sizes, alloc = [], torch.cuda.caching_allocator_alloc

    def counting(size, *args):
        sizes.append(size)
        return alloc(size, *args)

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", counting)
    cfg, ms = rt.rt_autotune(p, quad, order=order, integrator=rt.RT_HEUN, steps=1)
    builds = sum(s == -(-psi_bytes // 256) * 256 for s in sizes) // 2   # two buffers of psi each
    assert 11 <= builds <= most and (width == 16 or builds > 12)
    s = rt.Solver(p, quad, order=order, integrator=rt.RT_HEUN, **{k: cfg[k] for k in ("tile_x", "tile_y", "variant", "vec")})
    assert options(s) == (cfg["tile_x"], cfg["tile_y"], cfg["variant"], cfg["vec"])
    s.close()
