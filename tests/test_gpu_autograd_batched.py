"""Batched and repeated gradients of the field's training loss: the loss is a
scalar, so a batch of output gradients scales the one gradient."""
import pytest

import wost_inputs as wi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2410_18944_gb300 import api
    from test_gpu_streams import field_with_records
    F = field_with_records(api)
    p = wi.random_field_params(3, 3, [-1.1] * 3, [1.1] * 3, K=8, log2T=12, grid_scale=0.3)
    return F, [torch.tensor(p[k], dtype=torch.float32, device="cuda") for k in ("grid", "W1", "W2", "W3", "b3")]


def close(a, b):
    # the grid's gradient is an FP32 atomic sum: two runs differ in its order
    return float((a - b).abs().max()) <= 64 * 2.0 ** -24 * float(b.abs().max())


def test_batched_gradients(setup):
    import torch

    from paper_2410_18944_gb300.autograd import field_loss
    F, params = setup
    par = [t.clone().requires_grad_(True) for t in params]
    one = torch.autograd.grad(field_loss(F, *par), par)
    scale = torch.tensor([1.0, -2.0, 0.0, 0.5], device="cuda")
    many = torch.autograd.grad(field_loss(F, *par), par, grad_outputs=scale, is_grads_batched=True)
    for m, g in zip(many, one):
        assert m.shape == (4,) + g.shape
        for s, row in zip(scale.tolist(), m):
            assert close(row, s * g) if s else not row.any()


def test_vectorized_jacobian(setup):
    import torch

    from paper_2410_18944_gb300.autograd import field_loss
    F, params = setup
    want = torch.autograd.functional.jacobian(lambda *t: field_loss(F, *t), tuple(params))
    # (two equal outputs: the vectorised form takes a batch of output gradients)
    got = torch.autograd.functional.jacobian(lambda *t: field_loss(F, *t).expand(2), tuple(params), vectorize=True)
    for w, g in zip(want, got):
        assert g.shape == (2,) + w.shape and close(g[0], w) and close(g[1], w)
