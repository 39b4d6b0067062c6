"""Error reports of the three-dimensional step over nodes: a state that leaves
the EOS range in the last step is reported by the next call that waits."""
import numpy as np
import pytest

from paper_2205_00686_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("call", ["sync", "populations"])
def test_state_gone_bad_in_the_last_step_is_reported(call, prec):
    import paper_2205_00686_gb300 as lbm
    nx, ny, nz = 12, 6, 6
    # liquid at 0.86 T_c pressed together by the flow: psi^2 > 4.2 at t = 0, < 0
    # where one step takes the density above 9.1
    ux = np.broadcast_to(0.7 * np.sin(2 * np.pi * np.arange(nx) / nx), (nz, ny, nx)).copy()
    z = np.zeros_like(ux)
    fields = (np.full_like(z, 6.5), ux, z, z, np.full_like(z, 0.86 * W.TC))
    d = lbm.Domain3(nx, ny, nz, W.params(), W.periodic_bc3(), prec=prec)
    d.set_path(fused=False)
    d.init_fields(*fields)
    d.sync()
    d.step(1)
    with pytest.raises(lbm.LbmError) as e:
        getattr(d, call)()
    assert e.value.code == lbm.LBM_EPSI
    d.init_fields(*fields)
    d.sync()
    d.close()
