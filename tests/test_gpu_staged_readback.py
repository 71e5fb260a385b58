"""lb_get_fields between lb_stage_fields and lb_init_fields_staged: the fields of the run that is ending come back and the
staged ones of the next run stay as they were staged."""
import numpy as np
import pytest

from tests.test_gpu_staged_init import built, pinned, workload  # noqa: F401

pytestmark = pytest.mark.gpu


# the second size's copy of 16 MB is still under way when the steps and the read-back are enqueued
@pytest.mark.parametrize("n_cells,nx,ny", [(3, 64, 48), (2, 512, 512)])
@pytest.mark.parametrize("host", [pinned, np.array])
def test_fields_read_while_the_next_run_is_staged(n_cells, nx, ny, host):
    from paper_1004_5058_gb300 import Lattice
    cells, now = workload(n_cells, nx, ny, seed=5)
    then = [host(a) for a in workload(n_cells, nx, ny, seed=6)[1]]
    with Lattice(cells, "fp32") as a, Lattice(cells, "fp32") as b:
        b.init_fields(*now).step(3)
        want = b.fields()
        b.init_fields(*then).step(2)
        for _ in range(3):
            a.init_fields(*now).stage_fields(*then).step(3)
            got = a.fields()
            assert all(np.array_equal(x, y) for x, y in zip(got, want))
            a.init_fields_staged().step(2)
            assert np.array_equal(a.get_populations(), b.get_populations())
        a.init_fields(*now).step(3)  # nothing staged: the staging buffer serves both directions again
        assert all(np.array_equal(x, y) for x, y in zip(a.fields(), want))
