"""The many-steps-per-launch kernel of small lattices (LB_KERNEL_AUTO): equal to the tiled kernel bit for bit, the
sampled observables included (the same site arithmetic, the sums in the same order); on widths the tiled kernel does
not take, to the FP64 oracle and the generic kernel within rounding."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I
from tests._util import max_abs, oracle_runs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


def cells_of(nx, ny, bc, n, model):
    more = {"paper": {}, "two_tau": dict(tau=0.9, tau_b=1.2), "mrt": dict(s_nu=1.1, s_q=1.1), "forced": dict(f0=1e-4)}[model]
    return [I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405 - 0.02 * k, bc=bc, u_wall=0.01 * (k + 1), **more) for k in range(n)]


def run(cells, prec, kernel, pieces, sampling):
    from paper_1004_5058_gb300 import Lattice
    nx, ny, n = cells[0].nx, cells[0].ny, len(cells)
    ra, rb = I.random_fields(nx, ny, n_cells=n, seed=11)
    ux, uy = I.couette_velocity(nx, ny, 0.01, n_cells=n)
    with Lattice(cells, prec) as lat:
        if kernel == "tiled":  # with the tile that sets the order of auto's sums
            lat.set_kernel("auto")
            lat.set_kernel(*lat.kernel())
            assert lat.kernel()[0] == "tiled"
        else:
            lat.set_kernel(kernel)
        lat.init_fields(ra, rb, ux, uy).set_sampling(*sampling)
        launches = lat.kernel_launches
        for k in pieces:
            lat.step(k)
        obs = [lat.profile()[0]] + (list(lat.shear_stress()) if cells[0].bc else [])
        return lat.get_populations(), obs, lat.kernel_launches - launches, lat.profile()[1]


# widths and heights around the 32 x 8 patch; step counts around the 512 of a launch
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16", "fp16sr"])
@pytest.mark.parametrize("nx,ny,bc,n,model,pieces", [
    (64, 64, 1, 1, "paper", (1, 2, 7)), (32, 5, 0, 2, "forced", (9,)), (40, 9, 1, 3, "two_tau", (3, 6)),
    (72, 17, 0, 1, "mrt", (10,)), (320, 33, 1, 1, "paper", (8,)), (64, 16, 1, 2, "paper", (513, 2)),
    (256, 255, 1, 1, "paper", (4,)), (64, 64, 1, 15, "two_tau", (5,))])
def test_equals_tiled_kernel_bitwise(prec, nx, ny, bc, n, model, pieces):
    cells = cells_of(nx, ny, bc, n, model)
    fa, oa, la, na = run(cells, prec, "auto", pieces, (2, 3))
    fb, ob, lb, nb = run(cells, prec, "tiled", pieces, (2, 3))
    assert la < lb and na == nb
    assert np.array_equal(fa, fb)
    for a, b in zip(oa, ob):
        assert np.array_equal(a, b)


# any width: odd, narrower than a patch and its halo, one column into the next patch
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-13), ("fp32", 2e-6)])
@pytest.mark.parametrize("nx,ny,bc,model", [(5, 5, 0, "paper"), (7, 6, 1, "two_tau"), (33, 9, 0, "mrt"), (65, 10, 1, "paper"),
                                            (37, 23, 1, "mrt"), (101, 13, 0, "forced"), (129, 130, 1, "paper")])
def test_ragged_against_oracle(prec, tol, nx, ny, bc, model):
    cells = cells_of(nx, ny, bc, 2, model)
    f, obs, _, _ = run(cells, prec, "auto", (3, 17), (4, 5))
    ra, rb = I.random_fields(nx, ny, n_cells=2, seed=11)
    ux, uy = I.couette_velocity(nx, ny, 0.01, n_cells=2)
    for c, ref in enumerate(oracle_runs(cells, ra, rb, ux, uy, steps=20, sampling=(4, 5))):
        assert max_abs(f[c], ref.f) <= tol
    g, obs_g, _, _ = run(cells, prec, "generic", (20,), (4, 5))
    assert max_abs(f, g) <= tol
    for a, b in zip(obs, obs_g):
        assert max_abs(a, b) <= 10 * tol


def test_fp64_sizes_of_both_patches():
    for nx, ny in ((96, 106), (96, 107)):  # 10176 and 10272 sites: 8 x 4 and 16 x 8 patches
        cells = cells_of(nx, ny, 1, 1, "paper")
        a, _, _, _ = run(cells, "fp64", "auto", (12,), (0, 4))
        b, _, _, _ = run(cells, "fp64", "tiled", (12,), (0, 4))
        assert np.array_equal(a, b)


def test_reports_a_bad_density():
    from paper_1004_5058_gb300 import Lattice
    from paper_1004_5058_gb300 import _lib as L
    cells = cells_of(64, 64, 0, 1, "paper")
    ra, rb = I.random_fields(64, 64, seed=2)
    ra[0, 40, 33] = np.nan
    with Lattice(cells, "fp32") as lat:
        lat.init_fields(ra, rb).step(3)
        with pytest.raises(L.LBError) as e:
            lat.sync()
        assert e.value.status == L.LB_ERR_NONFINITE
        lat.init_fields(np.nan_to_num(ra, nan=0.6), rb).step(3).sync()


def test_autotune_keeps_state_and_may_pick_it(tmp_path):
    from paper_1004_5058_gb300 import Lattice
    cells = cells_of(64, 64, 1, 1, "paper")
    ra, rb = I.random_fields(64, 64, seed=2)
    cache = str(tmp_path / "tiles.txt")
    with Lattice(cells, "fp32") as lat, Lattice(cells, "fp32") as again:
        lat.init_fields(ra, rb).step(5)
        before = lat.get_populations()
        lat.autotune(cache)
        assert np.array_equal(before, lat.get_populations())
        again.init_fields(ra, rb)
        assert again.autotune(cache) == lat.kernel()
        n = again.kernel_launches
        again.step(100)
        assert again.kernel_launches - n <= 2  # one launch for all steps: the cached choice
