"""A small lattice whose cooperative launch is refused goes on with a launch per step (lb_test_inject 3 stands in for a
stream with too few SMs): the same populations and sums."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,nx,ny", [("fp32", 64, 48), ("fp64", 40, 33), ("fp32", 37, 23)])
def test_the_step_and_later_ones_go_on(prec, nx, ny):
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300._lib import LB_ERR_UNSUPPORTED
    cell = I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=1, u_wall=0.01)
    fields = I.random_fields(nx, ny, seed=3) + I.couette_velocity(nx, ny, 0.01)
    with Lattice([cell], prec) as a, Lattice([cell], prec) as b:
        for lat in (a, b):
            lat.init_fields(*fields).set_sampling(2, 3).step(7)
        assert a.lib.lb_test_inject(a.h, 3) == 0
        n = a.kernel_launches
        for k in (30, 11):
            a.step(k)
            b.step(k)
        assert a.kernel_launches - n >= 41  # one or two a step
        assert a.steps_done == b.steps_done == 48
        tol = 0.0 if a.kernel()[0] == "tiled" else 2e-6  # the generic pair adds in another order
        assert max_abs(a.get_populations(), b.get_populations()) <= tol
        assert max_abs(a.profile()[0], b.profile()[0]) <= tol and a.profile()[1] == b.profile()[1]
        a.set_kernel("auto")  # asks anew
        n = a.kernel_launches
        a.step(30)
        assert a.kernel_launches - n <= 3
        a.set_kernel("generic")
        assert a.lib.lb_test_inject(a.h, 3) == LB_ERR_UNSUPPORTED
