"""The FP64 kernels' psi outside the model's densities: at the end of its table (t = rho/rho0 = 64 ln2/16 = 2.77), where
1 - e^{-t} rounds to 1, at its clamp (t = 700), and NaN."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs, oracle_runs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("kernel", ["auto", "tiled", "generic"])  # auto: the patch kernel
@pytest.mark.parametrize("t", [1e-12, 2.7, 2.8, 40.0, 699.0, 701.0, 1e6])
def test_one_dense_site(kernel, t):
    from paper_1004_5058_gb300 import Lattice
    cell = I.make_cell("paper", nx=64, ny=32, g_ab=0.0)  # the pseudopotential forces alone
    ra, rb = I.random_fields(64, 32)
    ra[0, 11, 30] = rho = t * cell.rho0
    with Lattice([cell], "fp64") as lat:
        lat.set_kernel(kernel)
        f = lat.init_fields(ra, rb).step(1).get_populations()
    ref = oracle_runs([cell], ra, rb, steps=1)[0].f
    assert max_abs(f[0], ref) <= 1e-14 * (1.0 + rho)  # some ulp of the largest population


@pytest.mark.parametrize("kernel", ["auto", "tiled", "generic"])
def test_nan_is_reported(kernel):
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300._lib import LBError, LB_ERR_NONFINITE
    ra, rb = I.random_fields(64, 32)
    ra[0, 5, 7] = np.nan
    with Lattice([I.make_cell("paper", nx=64, ny=32)], "fp64") as lat:
        lat.set_kernel(kernel)
        with pytest.raises(LBError) as e:
            lat.init_fields(ra, rb).step(3).sync()
        assert e.value.status == LB_ERR_NONFINITE
