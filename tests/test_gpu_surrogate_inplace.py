"""mlp_forward with an output buffer inside its input buffer: every query's inputs are read before any output is written."""
import ctypes as C

import pytest

from tests.test_gpu_surrogate import box_and_inputs, env  # noqa: F401

pytestmark = pytest.mark.gpu


# one block of 32 queries, several, and more blocks than are resident at a time
@pytest.mark.parametrize("B", [3, 33, 4096, 30000])
@pytest.mark.parametrize("at", [0, 1, -1])  # outputs at the start, one float on, at the end of the inputs
def test_forward_over_its_inputs(env, B, at):  # noqa: F811
    torch, S = env
    from paper_1004_5058_gb300 import _lib as L
    box, x = box_and_inputs(S, B=B, seed=B)
    sg = S.Surrogate(box, sigma_scale=1.0, max_batch=B)
    sg.set_params(S.init_params(6))
    X = torch.tensor(x, dtype=torch.float32, device="cuda")
    want = sg.forward(X)
    first = at if at >= 0 else 5 * B - 2 * B
    flat = X.reshape(-1)
    L.check(sg.lib.mlp_forward(sg.h, C.c_void_p(X.data_ptr()), B, C.c_void_p(flat[first:].data_ptr())))
    assert torch.equal(flat[first:first + 2 * B].reshape(B, 2), want)
    sg.close()
