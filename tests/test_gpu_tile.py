"""Small-domain form of the step (several steps per launch over tiles of
nodes) against the sweep: a node's arithmetic is the same, so without buoyancy
the populations are equal bit for bit; with it the density sum is added in
another order and both agree to rounding (1e-12 in FP64; FP32 5e-5, a few
hundred roundings of 6e-8 after 41 steps).  Sizes sit at the edges of the
tiles and of the rounds of resident tiles."""
import numpy as np
import pytest

import parity as P
from paper_2205_00686_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def both(c, prec, chunks=(1, 40)):
    """Populations and step counts of the default path and of the sweep."""
    import paper_2205_00686_gb300 as lbm
    out = []
    for sweep in (False, True):
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
        if sweep:
            d.set_tile(128, 16)
        d.init_fields(*c.fields())
        for n in chunks:
            d.step(n)
        d.sync()
        out.append(d.populations() + (d.step_count,))
        d.close()
    return out


SIZES = [(2, 2), (9, 5), (32, 8), (33, 9), (65, 31), (97, 96), (300, 281)]


@pytest.mark.parametrize("prec", ["fp32", "fp64", "fp32_g16"])
@pytest.mark.parametrize("name", sorted(P.bc_variants()))
def test_equals_the_sweep_bit_for_bit(name, prec):
    for k, (nx, ny) in enumerate(SIZES):
        c = P.droplet_case(nx, ny, P.bc_variants()[name], seed=70 + k)
        if k % 3 == 2:     # general rates
            c.params = dict(c.params, s_e=1.1, s_eps=0.9, s_q=1.2, vs3=0.8, vs4=1.3)
        a, b = both(c, prec)
        assert a[3] == b[3] == 41
        for x, y in zip(a[:3], b[:3]):
            assert np.array_equal(x, y), (name, nx, ny, prec)


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 5e-5)])
@pytest.mark.parametrize("name", ["wall_open_heater", "two_walls_adiabatic", "open_dirichlet"])
def test_buoyancy_agrees_with_the_sweep(name, prec, tol):
    c = P.droplet_case(130, 70, P.bc_variants()[name], seed=5, gravity=3e-5)
    a, b = both(c, prec, chunks=(1, 39, 1))
    assert P.rel_err(a[0], b[0]) <= tol and P.rel_err(a[1], b[1]) <= tol
    one, many = both(c, prec, chunks=(41,))[0], a
    for x, y in zip(one[:3], many[:3]):
        assert np.array_equal(x, y)       # one launch or several: the same sums


@pytest.mark.parametrize("frozen", ["frozen_flow", "frozen_thermal"])
def test_frozen_lattices_equal_the_sweep(frozen):
    c = P.droplet_case(70, 45, P.bc_variants()["wall_open_heater"], seed=8)
    c.params = dict(c.params, **{frozen: 1})
    for x, y in zip(*both(c, "fp32")):
        assert np.array_equal(x, y)


def test_concurrent_small_domains_equal_their_solo_runs():
    """More grids than the GPU holds at once, on streams of their own: each
    launch waits until all of its tiles are resident, and every domain ends
    in its solo state."""
    import paper_2205_00686_gb300 as lbm
    specs = [("fp64", 64, 64), ("fp32", 256, 200), ("fp64", 120, 90), ("fp32_g16", 300, 170),
             ("fp32", 64, 64), ("fp64", 200, 200), ("fp32", 400, 333), ("fp64", 64, 64)]
    bc = P.bc_variants()["open_dirichlet"]
    cases = [P.droplet_case(nx, ny, bc, seed=90 + k) for k, (_, nx, ny) in enumerate(specs)]
    doms = []
    for (prec, nx, ny), c in zip(specs, cases):
        d = lbm.Domain(nx, ny, c.params, c.bc, prec=prec)
        d.init_fields(*c.fields())
        doms.append(d)
    for _ in range(4):
        for d in doms:
            d.step(300)
    for (prec, nx, ny), c, d in zip(specs, cases, doms):
        d.sync()
        s = lbm.Domain(nx, ny, c.params, c.bc, prec=prec)
        s.init_fields(*c.fields())
        s.step(1200)
        for x, y in zip(d.populations(), s.populations()):
            assert np.array_equal(x, y), (prec, nx, ny)
        s.close()
        d.close()


def test_target_stops_inside_a_launch():
    import paper_2205_00686_gb300 as lbm
    c = W.open_evaporation(90, 80, R=20.0)
    d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec="fp32")
    d.init_fields(*c.fields())
    d.set_target(37)
    d.step(100)
    assert d.step_count == 37
    a = d.populations()
    d.set_target(0)
    d.step(3)
    s = P.run_gpu(c, 37, "fp32")
    for x, y in zip(a, s.populations()):
        assert np.array_equal(x, y)
    s.step(3)
    for x, y in zip(d.populations(), s.populations()):
        assert np.array_equal(x, y)
