"""Steps enqueued while the caller captures the stream into a graph of its own: a small lattice takes a launch per step
there (no cooperative launch in the graph), a replay advances the state as often as it runs, and the handle steps on as
before afterwards."""
import numpy as np
import pytest

from paper_1004_5058_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("prec,kernel", [("fp32", "auto"), ("fp64", "auto"), ("fp32", "tiled"), ("fp32", "generic")])
def test_captured_steps(prec, kernel):
    import torch
    from paper_1004_5058_gb300 import Lattice
    nx, ny = 64, 48
    cell = I.make_cell("paper", nx=nx, ny=ny, g_ab=0.405, bc=1, u_wall=0.01)
    fields = I.random_fields(nx, ny, seed=3) + I.couette_velocity(nx, ny, 0.01)
    stream = torch.cuda.Stream()
    with Lattice([cell], prec, stream=stream) as a, Lattice([cell], prec) as b:
        a.set_kernel(kernel)
        b.set_kernel(kernel)
        a.init_fields(*fields).step(4).sync()
        b.init_fields(*fields).step(4)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            a.step(2)  # two steps: the populations are back in the buffer they came from
        for _ in range(3):
            with torch.cuda.stream(stream):
                graph.replay()
            b.step(2)
        assert np.array_equal(a.get_populations(), b.get_populations())
        a.step(9).step(5)
        b.step(9).step(5)
        assert np.array_equal(a.get_populations(), b.get_populations())
