"""The bounded waits of the many-steps kernel: with one flag withheld (lb_test_inject 4) every block gives up after its
bound, the batch reports a timeout, and a fresh state runs normally."""
import time

import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs, oracle_runs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


# one patch (it waits for itself), 4 x 6 patches, and more patches than resident blocks
@pytest.mark.parametrize("prec,nx,ny,n,tol", [("fp32", 32, 8, 1, 3e-6), ("fp32", 128, 48, 1, 3e-6), ("fp64", 40, 33, 1, 1e-12),
                                              ("fp64", 64, 64, 30, 1e-12)])
def test_withheld_flag_times_out_and_recovers(prec, nx, ny, n, tol):
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300._lib import LBError, LB_ERR_STATE, LB_ERR_TIMEOUT, LB_ERR_UNSUPPORTED
    cells = [I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=1, u_wall=0.01)] * n
    fields = I.random_fields(nx, ny, n_cells=n, seed=3) + I.couette_velocity(nx, ny, 0.01, n_cells=n)
    with Lattice(cells, prec) as lat:
        lat.init_fields(*fields).step(3).sync()
        assert lat.lib.lb_test_inject(lat.h, 4) == 0
        t0 = time.perf_counter()
        lat.step(700)  # two launches or more: the later ones see the flag of the first
        with pytest.raises(LBError) as e:
            lat.sync()
        waited = time.perf_counter() - t0
        assert e.value.status == LB_ERR_TIMEOUT
        assert 0.2 <= waited < 1.4, waited  # one bounded wait, not one per launch or patch
        with pytest.raises(LBError) as e:
            lat.step(1)
        assert e.value.status == LB_ERR_STATE
        lat.init_fields(*fields).step(10)
        ga, gb, _, _ = lat.fields()
        lat.set_kernel("generic")
        assert lat.lib.lb_test_inject(lat.h, 4) == LB_ERR_UNSUPPORTED
    (r,) = oracle_runs(cells[:1], *[f[:1] for f in fields], steps=10)
    oa, ob, _, _ = r.fields()
    assert max_abs(ga[0], oa) <= tol and max_abs(gb[0], ob) <= tol
