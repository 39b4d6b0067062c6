"""Region labelling at widths around its 32-column segments: a random vapour /
liquid pattern (percolating at 55 %, so regions wind through many segments and
seams) against the oracle's flood fill, label for label and statistic for
statistic."""
import numpy as np
import pytest

import oracle as O
from paper_2205_00686_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("nx,ny", [(2, 2), (31, 9), (32, 17), (33, 40), (64, 3), (97, 65), (300, 200)])
def test_random_pattern_matches_flood_fill(nx, ny, periodic):
    import paper_2205_00686_gb300 as lbm
    rg, rl = W.COEXISTENCE[0.86]
    thr = 0.5 * (rl + rg)
    rho = np.where(W.uniform(31 * nx + ny, nx * ny).reshape(ny, nx) < 0.55, 0.7, 5.5)
    c = W.static_droplet(nx, ny, R=1.0) if periodic else W.open_evaporation(nx, ny, R=1.0)
    z = np.zeros((ny, nx))
    d = lbm.Domain(nx, ny, c.params, c.bc, prec="fp32")
    d.init_fields(rho, z, z, np.full((ny, nx), 0.86 * W.TC))
    for below in (True, False):
        regs, lab = d.regions(thr, below=below, labels=True, max_regions=nx * ny)
        ol, oregs = O.components(rho, thr, below=below, periodic_x=periodic, periodic_y=periodic)
        assert np.array_equal(lab, ol)
        assert regs == oregs
    d.close()
