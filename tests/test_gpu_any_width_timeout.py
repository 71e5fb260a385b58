"""The tiled kernel's any-width form with a row whose copies are never issued (lb_test_inject 1): the waits run out after
their bound, the copies in flight (boxes and single words) are drained, and a fresh state runs normally."""
import time

import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("nx,ny,more", [(1021, 131, {}), (65, 2100, {}), (1022, 131, dict(s_nu=1.1))])
def test_stalled_copy_times_out_and_recovers(nx, ny, more):
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300._lib import LBError, LB_ERR_STATE, LB_ERR_TIMEOUT
    cell = I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=1, u_wall=0.01, **more)
    fields = I.random_fields(nx, ny, seed=3) + I.couette_velocity(nx, ny, 0.01)
    with Lattice([cell], "fp32") as lat, Lattice([cell], "fp32") as ref:
        assert lat.kernel()[0] == "generic"
        lat.init_fields(*fields).step(3).sync()
        assert lat.lib.lb_test_inject(lat.h, 1) == 0
        t0 = time.perf_counter()
        lat.step(40)  # one stalled launch, then 39 that see the flag and return
        with pytest.raises(LBError) as e:
            lat.sync()
        waited = time.perf_counter() - t0
        assert e.value.status == LB_ERR_TIMEOUT
        assert 1.5 <= waited < 10.0, waited  # one bounded wait, not one per launch
        with pytest.raises(LBError) as e:
            lat.step(1)
        assert e.value.status == LB_ERR_STATE
        lat.init_fields(*fields).step(20)
        ref.init_fields(*fields).step(20)
        assert max_abs(lat.get_populations(), ref.get_populations()) == 0.0
