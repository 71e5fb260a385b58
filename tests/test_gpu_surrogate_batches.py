"""Batch sizes at the edges of the surrogate kernels' work split: 32 queries per block (one or several per block over the
chip) for inference, slabs of 64 rows for the gradients.  Tolerances as in test_gpu_surrogate.py (BF16 products)."""
import numpy as np
import pytest

from tests.test_gpu_surrogate import box_and_inputs, env, oracle_params  # noqa: F401

pytestmark = pytest.mark.gpu


# 9728 = 2 blocks on each of 152 SMs, 32 queries each; beyond it a block takes a second group
@pytest.mark.parametrize("B", [1, 31, 32, 33, 9727, 9729, 19489])
def test_inference(env, B):  # noqa: F811
    torch, S = env
    from oracle import mlp
    box, x = box_and_inputs(S, B=B, seed=B)
    p = S.init_params(6)
    sg = S.Surrogate(box, sigma_scale=1.0, max_batch=B)
    sg.set_params(p)
    X = torch.tensor(x, dtype=torch.float32, device="cuda")
    out = sg.forward(X)
    stress, logit, _ = sg.serve(X)
    assert torch.equal(stress, out[:, 0]) and torch.equal(logit, out[:, 1])
    tail = sg.forward(X[-min(B, 17):].contiguous())  # a row's result does not depend on its place
    assert torch.equal(out[-min(B, 17):], tail)
    ref, _ = mlp.forward(oracle_params(p), mlp.normalise(x, box.center, box.half_range))
    whole, _ = mlp.forward(oracle_params(p), mlp.normalise(box_and_inputs(S, B=4096)[1], box.center, box.half_range))
    for c in range(2):
        scale = np.sqrt(np.mean(whole[:, c] ** 2))  # over the box, also for a batch of one
        assert np.max(np.abs(out[:, c].cpu().numpy() - ref[:, c])) <= 2e-2 * scale * (2 if B > 4096 else 1)
    sg.close()


@pytest.mark.parametrize("B", [1, 15, 63, 65, 129])
def test_gradients(env, B):  # noqa: F811
    torch, S = env
    from oracle import mlp
    box, x = box_and_inputs(S, B=B, seed=B)
    p = S.init_params(4)
    t, lab = 0.5 + np.sin(np.arange(B)), (np.arange(B) % 3 == 0).astype(np.float64)
    sg = S.Surrogate(box, sigma_scale=1.0, max_batch=256, lam=0.8)
    sg.set_params(p)
    g, loss = sg.gradients(*(torch.tensor(a, dtype=torch.float32, device="cuda") for a in (x, t, lab)))
    z = mlp.normalise(x, box.center, box.half_range)
    params = oracle_params(p)
    ref = mlp.flatten(mlp.gradients(params, z, t, lab, lam=0.8))
    assert loss == pytest.approx(mlp.loss(params, z, t, lab, lam=0.8), rel=2e-2)
    off = 0
    for (wo, wi), (bo,) in mlp.param_shapes():
        for n in (wo * wi, bo):
            a, r = g[off:off + n].astype(np.float64), ref[off:off + n]
            assert np.linalg.norm(a - r) <= 5e-2 * np.linalg.norm(r) + 1e-12, (off, n)
            off += n
    sg.close()
