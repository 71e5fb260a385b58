"""Launches of the many-steps kernel are short, so that other streams' kernels get their turn on the GPU."""
import time

import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,nx,ny,more", [("fp64", 320, 320, {}), ("fp64", 256, 256, dict(s_nu=1.1)), ("fp64", 64, 64, {}),
                                             ("fp32", 255, 256, {}), ("fp32", 64, 64, {}), ("fp16sr", 248, 256, {})])
def test_a_launch_lasts_milliseconds(prec, nx, ny, more):
    from paper_1004_5058_gb300 import Lattice
    ra, rb = I.random_fields(nx, ny, seed=2)
    with Lattice([I.make_cell("paper", nx=nx, ny=ny, **more)], prec) as lat:
        lat.init_fields(ra, rb).step(600).sync()
        n0, t0 = lat.kernel_launches, time.perf_counter()
        lat.step(600).sync()
        took, launches = time.perf_counter() - t0, lat.kernel_launches - n0
        assert launches < 600  # many steps each
        assert took / launches < 4e-3  # aimed at 2 ms
