"""Which kernel steps a lattice (lb_get_step_form), and a bench line that says nothing of a kernel that does not run."""
import pytest

from paper_1004_5058_gb300 import inputs as I
from tests.test_bench_contract import run_bench

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,nx,ny,form,kernel", [
    ("fp32", 64, 64, "patch", "tiled"), ("fp32", 37, 23, "patch", "generic"), ("fp64", 256, 256, "patch", "tiled"),
    ("fp16", 64, 64, "patch", "tiled"), ("fp16", 37, 23, "generic", "generic"), ("fp32", 256, 256, "tiled", "tiled"),
    ("fp32", 1021, 129, "tiled any width", "generic"), ("fp64", 1021, 129, "generic", "generic"),
    ("fp16sr", 1021, 129, "generic", "generic"), ("fp32", 45, 1500, "generic", "generic")])
def test_step_form(prec, nx, ny, form, kernel):
    from paper_1004_5058_gb300 import Lattice
    with Lattice([I.make_cell("paper", nx=nx, ny=ny)], prec) as lat:
        assert lat.step_form() == form and lat.kernel()[0] == kernel
        lat.init_fields(*I.random_fields(nx, ny))
        n = lat.kernel_launches
        lat.step(20)  # what the launches say: one for all steps, one a step, two a step
        assert lat.kernel_launches - n == {"patch": 1, "generic": 40}.get(form, 20)
        lat.set_kernel("generic")
        assert lat.step_form() == "generic"


@pytest.mark.parametrize("size,form", [(("64", "64"), "patch"), (("1021", "129"), "tiled any width"), (("256", "256"), "tiled")])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
def test_bench_line_describes_the_kernel_that_runs(prec, size, form):
    form = "generic" if (prec, form) == ("fp64", "tiled any width") else form
    kernel = ["--kernel", "tiled"] if form == "tiled" else []
    d = run_bench("--steps", "3", "--warmup", "3", "--nx", size[0], "--ny", size[1], "--cells", "1", "--chunk", "20",
                  "--precision", prec, "--no-cpu-baseline", "--bvp-steps", "0", *kernel)
    rf, cfg = d["roofline"], d["config"]
    if form in ("patch", "tiled any width") and cfg["step_form"] != form:
        pytest.skip("the tuner chose %s" % cfg["step_form"])
    assert (cfg["launch"] is not None) == (cfg["step_form"] == "tiled")
    if cfg["step_form"] != "tiled":
        assert rf["traffic"] is None
    if prec == "fp64":
        assert (rf["frac"] is not None) == (cfg["step_form"] == "tiled")
    else:  # bytes and time of the same number of steps
        assert rf["algorithmic_bytes_per_launch"] / rf["mean_launch_ms"] * 1e-6 == pytest.approx(rf["achieved"], rel=1e-9)
        assert rf["algorithmic_bytes_per_launch"] == pytest.approx(144 * int(size[0]) * int(size[1]) * rf["steps_per_launch"])
