"""Arrays that are used on another stream than the call's."""
import ctypes as C

import numpy as np
import pytest

import wost_inputs as wi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2410_18944_gb300 import api as A
    return A


def field_with_records(api, dim=3, n=500):
    lo, hi = [-1.1] * dim, [1.1] * dim
    p = wi.random_field_params(dim, 3, lo, hi, K=8, log2T=12, grid_scale=0.3)
    F = api.Field(dim, lo, hi, log2_table=12)
    F.set_params(**{k: p[k] for k in ("grid", "W1", "W2", "W3", "b3")})
    r = np.random.default_rng(5)
    rec = np.zeros((n, 12), np.float32)
    rec[:, :dim] = r.uniform(-1, 1, (n, dim))
    nu = r.normal(size=(n, dim))
    rec[:, 3:3 + dim] = nu / np.linalg.norm(nu, axis=1, keepdims=True)
    rec[:, 10] = 0.2
    rec[:, 11] = r.uniform(0, 1, n)
    F.set_records(rec)
    return F


def test_gradient_array_written_on_the_default_stream(api):
    """A gradient array that the default stream is still filling when the call
    starts on another stream ends up with the gradient."""
    import torch

    from paper_2410_18944_gb300 import _lib as L
    F = field_with_records(api)
    _, g = F.train_grad()
    out = torch.empty(g["grid"].shape, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)   # about 50 ms
    out.fill_(7.0)
    lib, loss, null = L.load(), C.c_float(), C.cast(None, L._fp)
    e = api.exec_defaults(stream=side)
    L.check(lib.wost_train_grad(F._h, C.byref(e), C.byref(loss), C.cast(C.c_void_p(out.data_ptr()), L._fp), null, null,
                                null, null))
    torch.cuda.synchronize()
    # (two orders of FP32 atomic sums, as in test_gpu_paths)
    assert np.abs(out.cpu().numpy() - g["grid"]).max() <= 64 * 2.0 ** -24 * np.abs(g["grid"]).max()
