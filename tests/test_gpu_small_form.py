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
