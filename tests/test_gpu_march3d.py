"""The 3-D step's forms (marching tiles and kernels over the nodes) at unit and
at general relaxation rates against the FP64 oracle: 1e-10 on fields, 1e-12 on
populations after 20 steps, at sizes that end inside a 32 x 8 tile, on it and
one past it, with walls, buoyancy and every segment remainder."""
import numpy as np
import pytest

import oracle as O
import parity as P
from paper_2205_00686_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


def case(nx, ny, nz, walls, general):
    p = W.params(gravity=2e-5)
    if general:
        p.update(s_e=1.1, s_eps=0.9, s_q=1.2, vs3=0.8, vs4=1.3)
    c = W.droplet3d(nx, ny, nz, R=0.3 * min(nx, ny, nz), amp=1e-3, p=p)
    z, y, x = np.mgrid[0:nz, 0:ny, 0:nx].astype(float)
    c.T = c.T * (1.0 + 0.02 * np.exp(-((x - 0.3 * nx) ** 2 + (y - 0.6 * ny) ** 2) / 20.0))
    if walls:
        c.bc = W.wall_bc3(0.95 * W.TC, 0.88 * W.TC, theta_deg=70.0)
    return c


@pytest.mark.parametrize("fused,zseg", [(True, 0), (True, 4), (False, 0)])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("shape", [(32, 8, 9), (33, 9, 10), (31, 17, 12)])
def test_fp64_matches_oracle(shape, general, walls, fused, zseg):
    import paper_2205_00686_gb300 as lbm
    c = case(*shape, walls, general)
    o = O.Sim3(c.nx, c.ny, c.nz, c.params, c.bc)
    o.init(*c.fields())
    o.step(20)
    d = lbm.Domain3(c.nx, c.ny, c.nz, c.params, c.bc, prec="fp64")
    d.set_path(fused, zseg)
    d.init_fields(*c.fields())
    d.step(20)
    for a, b in zip(d.get_fields(), o.fields()):
        assert P.rel_err(a, b) <= 1e-10
    for a, b in zip(d.populations()[:2], o.populations()[:2]):
        assert P.rel_err(a, b) <= 1e-12
    d.close()


@pytest.mark.parametrize("general", [False, True])
def test_fp32_forms_agree(general):
    """FP32: the two forms contract their operations differently; after 10
    steps the populations agree to 10 x 2^-22 of their largest value."""
    import paper_2205_00686_gb300 as lbm
    c = case(45, 21, 19, True, general)
    out = []
    for fused in (True, False):
        d = lbm.Domain3(c.nx, c.ny, c.nz, c.params, c.bc, prec="fp32")
        d.set_path(fused, 0)
        d.init_fields(*c.fields())
        d.step(10)
        out.append(d.populations())
        d.close()
    for a, b in zip(out[0][:2], out[1][:2]):
        assert P.rel_err(a, b) <= 10.0 * 2.0 ** -22
