"""With buoyancy every step reads the mean density of the step before.  Its sum
is exact (fixed-point numbers added as integers), so a domain's state does not
depend on how it is cut: alone in any tile, by the small-domain form, or in a
batch whatever its other members are, the populations are equal bit for bit."""
import numpy as np
import pytest

import parity as P

pytestmark = pytest.mark.gpu

STEPS = 41


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def domain(c, prec):
    import paper_2205_00686_gb300 as lbm
    d = lbm.Domain(c.nx, c.ny, c.params, c.bc, prec=prec)
    d.init_fields(*c.fields())
    return d


def solo(c, prec, tile=None, staged=None):
    d = domain(c, prec)
    if tile:
        d.set_tile(*tile)
    if staged is not None:
        d.staged = staged
    d.step(STEPS)
    assert bool(d.small_form()[0]) == (tile is None and staged is None)
    d.sync()
    out = d.populations()
    d.close()
    return out


def in_batch(cases, prec):
    """Populations of the first case as a member of an untuned batch."""
    import paper_2205_00686_gb300 as lbm
    b = lbm.Batch()
    doms = [domain(c, prec) for c in cases]
    for d in doms:
        b.attach(d)
    b.step(STEPS)
    assert b.sync() == 0
    rows = b.tile()[1]
    b.detach(doms[0])
    out = doms[0].populations()
    b.close()
    for d in doms:
        d.close()
    return out, rows


@pytest.mark.parametrize("prec", ["fp32", "fp64", "fp32_g16"])
@pytest.mark.parametrize("name", ["wall_open_heater", "two_walls_adiabatic"])
def test_state_does_not_depend_on_the_cut(name, prec):
    v = P.bc_variants()
    c = P.droplet_case(130, 203, v[name], seed=61, gravity=3e-5)
    others = [P.droplet_case(nx, ny, v[name], seed=62 + k, gravity=3e-5)
              for k, (nx, ny) in enumerate([(600, 611), (900, 700), (500, 400)])]
    ref = solo(c, prec, tile=(128, 64))
    few, rows_few = in_batch([c], prec)
    many, rows_many = in_batch([c] + others, prec)
    assert rows_few != rows_many
    runs = {"small form": solo(c, prec), "13 rows": solo(c, prec, tile=(128, 13)),
            "one segment": solo(c, prec, tile=(256, 203)), "batch of one": few, "batch of four": many}
    for how, got in runs.items():
        for a, b in zip(got, ref):
            assert np.array_equal(a, b), how


def test_staged_rows_sum_the_same():
    c = P.droplet_case(230, 150, P.bc_variants()["open_dirichlet"], seed=66, gravity=3e-5)
    ref = solo(c, "fp32", tile=(128, 37))
    for a, b in zip(solo(c, "fp32", staged=True), ref):
        assert np.array_equal(a, b)
    for a, b in zip(solo(c, "fp32"), ref):
        assert np.array_equal(a, b)
