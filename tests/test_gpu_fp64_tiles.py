"""Tile and segment height of FP64 lattices whose width is a multiple of 32 and of no wider tile."""
import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


# shapes on which a wider tile, or the heights of a model that takes every row to fill the FP64 pipe, took at least 1.15
# times as long
@pytest.mark.parametrize("nx,ny,n", [(96, 96, 64), (96, 64, 400), (160, 160, 32), (160, 300, 12), (160, 512, 4), (224, 224, 16), (480, 1000, 2)])
def test_narrow_tiles_that_use_the_whole_pipe(nx, ny, n):
    from paper_1004_5058_gb300 import Lattice
    cells = [I.make_cell("paper", nx=nx, ny=ny, bc=1)] * n
    with Lattice(cells, "fp64") as lat, Lattice(cells, "fp64", slab=(0, ny // 2)) as slab:
        kind, tx, ty = lat.kernel()
        assert (kind, tx) == ("tiled", 32) and slab.kernel()[:2] == ("tiled", 32)  # the order of the sums is the tile's
        items = (nx // 32) * -(-ny // ty) * n
        per_sm = -(-items // 152)
        assert per_sm >= 3  # one column warp each, on the SM's four sub-partitions


def test_other_widths_and_precisions_keep_theirs():
    from paper_1004_5058_gb300 import Lattice
    for prec, nx, tile in (("fp64", 128, 128), ("fp64", 192, 64), ("fp64", 200, 128), ("fp32", 160, 128), ("fp32", 96, 64), ("fp64", 32, 32)):
        with Lattice([I.make_cell("paper", nx=nx, ny=700)] * 4, prec) as lat:
            assert lat.kernel()[:2] == ("tiled", tile)
