"""Large lattices of a width the tiled kernel's halo boxes cannot serve (odd, or rows that are no multiple of 16 bytes):
LB_KERNEL_AUTO runs the tiled kernel's any-width form, checked here against the generic kernel pair."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def run(cells, prec, kernel, steps, sampling):
    from paper_1004_5058_gb300 import Lattice
    nx, ny, n = cells[0].nx, cells[0].ny, len(cells)
    ra, rb = I.random_fields(nx, ny, n_cells=n, seed=11)
    ux, uy = I.couette_velocity(nx, ny, 0.01, n_cells=n)
    with Lattice(cells, prec) as lat:
        assert lat.kernel()[0] == "generic"
        lat.set_kernel(kernel)
        lat.init_fields(ra, rb, ux, uy).set_sampling(*sampling)
        n0 = lat.kernel_launches
        lat.step(steps)
        obs = [lat.profile()[0]] + (list(lat.shear_stress()) if cells[0].bc else [])
        return lat.get_populations(), obs, lat.kernel_launches - n0


# one column and one pair more or less than strips of 128 and 64; widths whose last halo word or 16-byte group is split
SHAPES = [(65, 2100), (127, 1040), (129, 1021), (130, 1009), (191, 700), (1021, 129), (1022, 131), (254, 517)]


@pytest.mark.parametrize("nx,ny", SHAPES)
@pytest.mark.parametrize("bc,model", [(0, {}), (1, {}), (1, dict(tau=0.9, tau_b=1.2)), (0, dict(f0=1e-4)), (1, dict(s_nu=1.1, s_q=1.1))])
def test_fp32_against_generic(nx, ny, bc, model):
    cells = [I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=bc, u_wall=0.01, **model)]
    fa, oa, la = run(cells, "fp32", "auto", 20, (4, 5))
    fb, ob, lb = run(cells, "fp32", "generic", 20, (4, 5))
    assert la < lb
    assert max_abs(fa, fb) <= 2e-6  # 20 steps of FP32 roundings (6e-8 of f < 0.5 each), both sides
    for a, b in zip(oa, ob):
        assert max_abs(a, b) <= 2e-6


@pytest.mark.parametrize("prec,ulp", [("fp16", 2.0 ** -10), ("fp16sr", 2.0 ** -9)])
@pytest.mark.parametrize("nx,ny", [(65, 2100), (129, 1021), (1012, 131), (1021, 129)])
def test_fp16_one_step_against_generic(prec, ulp, nx, ny):
    cells = [I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=1, u_wall=0.01)]
    fa, _, _ = run(cells, prec, "auto", 1, (0, 0))
    fb, _, _ = run(cells, prec, "generic", 1, (0, 0))
    # |g| = |f - w rho_bar| < 0.06 here, stored to an ulp on each side
    assert max_abs(fa, fb) <= ulp * 0.0625


def test_batch_of_odd_cells():
    cells = [I.make_cell("paper", nx=101, ny=260, g_ab=0.4 - 0.01 * k, bc=1, u_wall=0.001 * k) for k in range(6)]
    fa, oa, _ = run(cells, "fp32", "auto", 20, (4, 5))
    fb, ob, _ = run(cells, "fp32", "generic", 20, (4, 5))
    assert max_abs(fa, fb) <= 2e-6
    for a, b in zip(oa, ob):
        assert max_abs(a, b) <= 2e-6


def test_explicit_choices_are_as_before():
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300._lib import LBError, LB_ERR_UNSUPPORTED
    with Lattice([I.make_cell("paper", nx=1021, ny=129, bc=1)], "fp32") as lat:
        with pytest.raises(LBError) as e:
            lat.set_kernel("tiled", 128, 0)
        assert e.value.status == LB_ERR_UNSUPPORTED
        assert lat.kernel() == ("generic", 32, 8) and lat.launch_shape() is None


def test_reports_a_bad_density_in_the_last_odd_column():
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300 import _lib as L
    ra, rb = I.random_fields(1021, 131, seed=2)
    with Lattice([I.make_cell("paper", nx=1021, ny=131, bc=0)], "fp32") as lat:
        lat.init_fields(ra, rb).step(3).sync()
        ra[0, 70, 1020] = np.nan
        lat.init_fields(ra, rb).step(1)
        with pytest.raises(L.LBError) as e:
            lat.sync()
        assert e.value.status == L.LB_ERR_NONFINITE
