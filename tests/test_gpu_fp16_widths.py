"""FP16 storage of widths the tiled kernel does not take runs the generic kernel pair under LB_KERNEL_AUTO, small lattices
and large ones: the FP32 sums before a rounding to FP16, and the dither of its storage, are those of that kernel."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


# odd, rows of no whole 16 bytes, narrower than the narrowest tile; below and above 2^16 sites
@pytest.mark.parametrize("prec", ["fp16", "fp16sr"])
@pytest.mark.parametrize("nx,ny,bc,model", [(37, 23, 1, {}), (24, 40, 0, {}), (100, 31, 1, dict(tau_b=0.9)), (129, 510, 1, {}),
                                            (1021, 129, 0, dict(f0=1e-4)), (1012, 131, 1, dict(s_nu=1.1))])
def test_auto_is_the_generic_pair(prec, nx, ny, bc, model):
    from paper_1004_5058_gb300 import Lattice
    cell = I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=bc, u_wall=0.01, **model)
    fields = I.random_fields(nx, ny, seed=11) + I.couette_velocity(nx, ny, 0.01)
    got = []
    for kernel in ("auto", "generic"):
        with Lattice([cell], prec) as lat:
            assert lat.kernel()[0] == "generic"
            lat.set_kernel(kernel)
            lat.init_fields(*fields).set_sampling(2, 3).step(12)
            got.append((lat.get_populations(), lat.profile()[0]))
    for a, b in zip(*got):
        assert np.array_equal(a, b)
