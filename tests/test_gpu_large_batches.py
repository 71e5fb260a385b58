"""FP32 batches whose two buffers are more than twice the L2 run the tiled kernel's form for lattices that stream from
memory: every cell of such a batch equals the same cell simulated alone, which runs the form for smaller lattices."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def run(cells, fields):
    from paper_1004_5058_gb300 import Lattice
    with Lattice(cells, "fp32") as lat:
        assert lat.kernel()[:2] == ("tiled", 128)
        lat.init_fields(*fields).set_sampling(3, 4)
        lat.step(11)
        return lat.get_populations(), lat.profile()[0]


# both buffers hold 2 x 18 x 4 bytes per site: 256 MB are 1.864e6 sites; the sizes lie just above, in whole strips
@pytest.mark.parametrize("bc,f0", [(1, 0.0), (0, 1e-5)])
@pytest.mark.parametrize("nx,ny", [(1024, 911), (1152, 811), (128, 7283)])
def test_cells_of_a_large_batch_equal_single_cells(nx, ny, bc, f0):
    cells = [I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405 - 0.02 * k, bc=bc, u_wall=0.01, f0=f0) for k in range(2)]
    fields = I.random_fields(nx, ny, n_cells=2, seed=5) + I.couette_velocity(nx, ny, 0.01, n_cells=2)
    pops, prof = run(cells, fields)
    pops, prof = pops.reshape(2, -1), prof.reshape(2, -1)
    for k in range(2):
        f1, p1 = run(cells[k:k + 1], [np.ascontiguousarray(a[k:k + 1]) for a in fields])
        assert np.array_equal(pops[k], f1.reshape(-1))  # the same operations on the same values: no tolerance
        assert np.max(np.abs(prof[k] - p1.reshape(-1))) <= 1e-12  # sums of 1152 speeds below 0.1, in FP64
