"""The forward pass and the served values against the same network in plain torch that rounds where the kernel does: the
normalised inputs, the weights and each layer's activations to BF16, bias and tanh in FP32, products summed in 64 bits.

What may differ is the FP32 summation (128 terms of at most 0.09: below 1e-6) and, where a sum lies that near a rounding
boundary, one BF16 step of an activation: 2^-8 times a weight of at most 128^-1/2, 3.5e-4 in what follows.  A boundary is
that near for some 2e-4 of the 384 activations of a query, so at least three queries of four have none; six steps at once
bound the others."""
import numpy as np
import pytest

from tests.test_gpu_surrogate import box_and_inputs, env  # noqa: F401

pytestmark = pytest.mark.gpu


def plain(torch, box, p, x):
    from oracle import mlp
    r = lambda a: a.to(torch.bfloat16)  # noqa: E731
    f32 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")  # noqa: E731
    h, off = r((x - f32(box.center)) / f32(box.half_range)), 0
    shapes = mlp.param_shapes()
    for l, ((o, i), _) in enumerate(shapes):
        W, b = f32(p[off:off + o * i]).reshape(o, i), f32(p[off + o * i:off + o * i + o])
        off += o * i + o
        y = (h.double() @ r(W).double().T).float() + b
        h = r(torch.tanh(y)) if l + 1 < len(shapes) else y
    return h


@pytest.mark.parametrize("B", [1, 33, 300, 10000])
def test_rounding_by_rounding(env, B):  # noqa: F811
    torch, S = env
    box, x = box_and_inputs(S, B=max(B, 64), seed=B)
    p = S.init_params(7)
    assert np.abs(p).max() <= 0.5
    X = torch.tensor(x, dtype=torch.float32, device="cuda")
    sg = S.Surrogate(box, sigma_scale=1.0, max_batch=max(B, 64))
    sg.set_params(p)
    ref = plain(torch, box, p, X)
    got = torch.cat([sg.forward(X[k:k + B].contiguous()) for k in range(0, len(X), B)])  # single queries too
    stress, logit, _ = sg.serve(X)
    for a in (got, torch.stack([stress, logit], 1)):
        far = (a - ref).abs().amax(1)
        assert float(far.quantile(0.75)) <= 1e-5
        assert float(far.max()) <= 6 * 3.5e-4
    sg.close()
