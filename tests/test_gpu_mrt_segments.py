"""The segment height of cells with multiple relaxation times follows from the CTAs that their kernel has resident: no
launch leaves most of its last round empty."""
import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec", ["fp32", "fp16", "fp16sr"])
@pytest.mark.parametrize("nx,ny,n", [(96, 512, 16), (64, 512, 20), (192, 400, 8), (320, 320, 8)])
def test_rounds_are_full(prec, nx, ny, n):
    from paper_1004_5058_gb300 import Lattice
    with Lattice([I.make_cell("paper", nx=nx, ny=ny, bc=1, s_nu=1.1)] * n, prec) as lat:
        _, tx, ty = lat.kernel()
        items, ctas = -(-nx // tx) * -(-ny // ty) * n, lat.launch_shape()[0]
        assert items / (-(-items // ctas) * ctas) >= 0.8  # 0.6 with the heights of the BGK kernel's occupancy
