"""Choice and failure paths of the small-domain form of the step."""
import numpy as np
import pytest

import parity as P

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("prec", ["fp32", "fp64", "fp32_g16"])
def test_refused_cooperative_launch_goes_on_with_the_sweep(prec):
    """A device that refuses the cooperative launch (answered by the test hook
    on the host) costs the context the small-domain form and nothing else."""
    import paper_2205_00686_gb300 as lbm
    c = P.droplet_case(130, 70, P.bc_variants()["open_dirichlet"], seed=31)
    ref = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
    ref.init_fields(*c.fields())
    d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
    d.init_fields(*c.fields())
    d.step(5)
    assert d.small_form()[0] > 0
    d.set_wait_probe(2)
    d.step(40)
    assert d.small_form() == (0, 0, 0, 0)
    d.set_wait_probe(0)
    d.step(3)
    ref.step(48)
    assert ref.small_form()[0] > 0
    assert d.step_count == ref.step_count == 48
    for a, b in zip(d.populations(), ref.populations()):
        assert np.array_equal(a, b)
    ref.close()
    d.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_rates_changed_after_the_plan(prec):
    """The plan is made at creation; lbm_reconfigure may then switch between
    unit and general rates, another kernel on the same grid.  A domain of
    several rounds of tiles keeps agreeing with the sweep."""
    import paper_2205_00686_gb300 as lbm
    c = P.droplet_case(430, 410, P.bc_variants()["open_dirichlet"], seed=32)
    general = dict(c.params, s_e=1.1, s_eps=0.9, s_q=1.2, vs3=0.8, vs4=1.3)
    pops = []
    for sweep in (False, True):
        d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
        if sweep:
            d.set_tile(128, 32)
        d.init_fields(*c.fields())
        d.step(7)
        d.reconfigure(general, c.bc)
        d.step(7)
        tx, ty, tiles, ctas = d.small_form()
        assert (tx > 0) != sweep and (sweep or tiles > ctas)
        d.reconfigure(c.params, c.bc)
        d.step(7)
        d.sync()
        pops.append(d.populations())
        d.close()
    for a, b in zip(*pops):
        assert np.array_equal(a, b)


def test_autotune_keeps_no_form_that_was_refused():
    """A trial whose launch is refused is out of the comparison, and what the
    autotuner learned for one set of boundaries and rates says nothing about
    another."""
    import paper_2205_00686_gb300 as lbm
    v = P.bc_variants()
    c = P.droplet_case(210, 150, v["open_dirichlet"], seed=33)

    def fresh(bc="open_dirichlet", **over):
        return lbm.Domain(c.nx, c.ny, dict(c.params, **over), v[bc], prec="fp32")

    d = fresh()
    d.init_fields(*c.fields())
    d.set_wait_probe(2)
    d.autotune(4)
    assert d.small_form() == (0, 0, 0, 0)
    assert fresh().small_form() == (0, 0, 0, 0)
    assert fresh("two_walls_adiabatic").small_form()[0] > 0
    assert fresh(s_q=1.2).small_form()[0] > 0
    d.set_wait_probe(0)
    d.autotune(4)
    assert d.small_form()[0] > 0 and fresh().small_form() == d.small_form()
    d.close()


TILES = {"fp32": [(8, 8), (32, 8), (32, 10), (32, 12)],
         "fp64": [(8, 4), (8, 8), (16, 8), (32, 8), (20, 14)]}
TILES["fp32_g16"] = TILES["fp32"]


@pytest.mark.parametrize("prec,tx,ty", [(p, *t) for p in TILES for t in TILES[p]])
@pytest.mark.parametrize("name", ["wall_open_heater", "open_dirichlet", "periodic_flow_fixed_T"])
def test_every_tile_equals_the_sweep(name, prec, tx, ty):
    """Whichever tile the plan takes: domains smaller than a tile, with ragged
    last tiles, one tile past 152 (a round of one CTA per SM) and past 304."""
    import paper_2205_00686_gb300 as lbm
    sizes = [(3, 2), (tx + 1, 2 * ty - 1), (9 * tx - 3, 17 * ty - 1), (5 * tx - 1, 61 * ty - 2)]
    for k, (nx, ny) in enumerate(sizes):
        c = P.droplet_case(nx, ny, P.bc_variants()[name], seed=40 + k, gravity=3e-5)
        if k % 2:     # general rates
            c.params = dict(c.params, s_e=1.1, s_eps=0.9, s_q=1.2, vs3=0.8, vs4=1.3)
        pops = []
        for sweep in (False, True):
            d = lbm.Domain(nx, ny, c.params, c.bc, prec=prec)
            if sweep:
                d.set_tile(128, 16)
            else:
                d.set_small_form(tx, ty)
                assert d.small_form()[:3] == (tx, ty, -(-nx // tx) * -(-ny // ty))
            d.init_fields(*c.fields())
            d.step(1)
            d.step(20)
            d.sync()
            assert d.step_count == 21
            assert bool(d.small_form()[0]) != sweep
            pops.append(d.populations())
            d.close()
        for a, b in zip(*pops):
            assert np.array_equal(a, b), (nx, ny)


def test_tile_selection():
    import paper_2205_00686_gb300 as lbm
    c = P.droplet_case(300, 200, P.bc_variants()["open_dirichlet"])
    d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec="fp32")
    own = d.small_form()
    assert own[0] > 0 and 0 < own[3] <= own[2]
    for bad in [(7, 7), (20, 14), (32, 9)]:
        with pytest.raises(lbm.LbmError) as e:
            d.set_small_form(*bad)
        assert e.value.code == lbm.LBM_EINVAL
        assert d.small_form() == own
    d.set_tile(128, 16)
    assert d.small_form() == (0, 0, 0, 0)
    d.set_small_form()
    assert d.small_form() == own
    d.close()
    big = lbm.Domain(1100, 1000, c.params, c.bc, prec="fp32")
    big.set_small_form()
    assert big.small_form() == (0, 0, 0, 0)
    with pytest.raises(lbm.LbmError):
        big.set_small_form(32, 8)
    big.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_grid_barrier_timeout_is_reported_and_cleared(prec):
    """With the test hook on, a CTA that finds the grid barrier incomplete gives
    up: LBM_ETIMEOUT is reported, nothing hangs (3000 steps are three launches,
    of which the later ones leave at once), and a fresh state steps normally.  One
    step has no barrier and is unaffected."""
    import time

    import paper_2205_00686_gb300 as lbm
    c = P.droplet_case(130, 170, P.bc_variants()["wall_open_heater"], seed=35, gravity=3e-5)
    ref = P.run_gpu(c, 41, prec)
    d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
    d.init_fields(*c.fields())
    d.set_wait_probe(1)
    d.step(1)
    d.sync()
    t0 = time.perf_counter()
    d.step(3000)
    with pytest.raises(lbm.LbmError) as e:
        d.sync()
    assert e.value.code == lbm.LBM_ETIMEOUT
    assert time.perf_counter() - t0 < 10.0
    with pytest.raises(lbm.LbmError) as e:
        d.step(1)
    assert e.value.code == lbm.LBM_ETIMEOUT
    d.set_wait_probe(0)
    d.init_fields(*c.fields())
    d.step(41)
    d.sync()
    assert d.small_form()[0] > 0 and d.step_count == 41
    for a, b in zip(d.populations(), ref.populations()):
        assert np.array_equal(a, b)
    d.close()
