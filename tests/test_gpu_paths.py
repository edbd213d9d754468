"""Branches of the launch and copy paths: each against the general one."""
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


def _params(dim, K, seed=3, grid_type=0, **kw):
    lo, hi = [-1.1] * dim, [1.1] * dim
    p = wi.random_field_params(dim, seed, lo, hi, K=K, log2T=12, grid_scale=0.3, grid_type=grid_type, **kw)
    return lo, hi, {k: np.ascontiguousarray(p[k], np.float32) for k in ("grid", "W1", "W2", "W3", "b3")}


@pytest.mark.parametrize("dim,K", [(2, 8), (3, 8), (3, 3), (2, 16), (3, 16)])
def test_decode_of_ragged_sizes(api, dim, K):
    """Rows are staged per warp: every size gives the rows of the whole set."""
    lo, hi, p = _params(dim, K)
    F = api.Field(dim, lo, hi, K=K, log2_table=12)
    F.set_params(**p)
    x = np.random.default_rng(1).uniform(-1, 1, (700, dim))
    whole = F.decode(x)
    assert np.isfinite(whole).all()
    for n in (1, 23, 25, 31, 33, 127, 129, 255, 257, 513):
        assert np.array_equal(F.decode(x[:n]), whole[:n]), n


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("offset", [0, 1])
def test_set_params_from_device_arrays(api, dim, offset):
    """One pass over device arrays (16-byte aligned, or copied when not) loads
    what the host arrays load, and clears the Adam state."""
    import torch

    from paper_2410_18944_gb300 import _lib as L
    lo, hi, p = _params(dim, 8)
    A, B = (api.Field(dim, lo, hi, log2_table=12) for _ in range(2))
    A.set_params(**p)
    dev = []
    for k in ("grid", "W1", "W2", "W3", "b3"):
        buf = torch.empty(p[k].size + offset, device="cuda")
        buf[offset:].copy_(torch.tensor(p[k].ravel()))
        dev.append(buf[offset:])
    torch.cuda.synchronize()
    ptr = [C.cast(C.c_void_p(t.data_ptr()), L._fp) for t in dev]
    assert L.load().wost_field_set_params(B._h, *ptr) == 0
    for k, v in B.get_params().items():
        assert np.array_equal(v, p[k]), k
    x = np.random.default_rng(1).uniform(-1, 1, (300, dim))
    assert np.array_equal(A.decode(x), B.decode(x))


@pytest.mark.parametrize("dim", [2, 3])
def test_grid_gradient_in_place(api, dim):
    """The gradient accumulated in a device array is the one copied to the
    host, up to the order of its FP32 atomic sums: at most n adds of a value
    each round by 2^-24 of the sum of magnitudes, here bounded by 64 x 2^-24 of
    the largest entry."""
    import torch

    from paper_2410_18944_gb300 import _lib as L
    from paper_2410_18944_gb300.autograd import _exec
    lo, hi, p = _params(dim, 8)
    F = api.Field(dim, lo, hi, log2_table=12)
    F.set_params(**p)
    r = np.random.default_rng(5)
    n = 500
    rec = np.zeros((n, 12), np.float32)
    rec[:, :dim] = r.uniform(-1, 1, (n, dim))
    nu = r.normal(size=(n, dim))
    rec[:, 3:3 + dim] = nu / np.linalg.norm(nu, axis=1, keepdims=True)
    rec[:, 10] = 0.2
    rec[:, 11] = r.uniform(0, 1, n)
    F.set_records(rec)
    loss, g = F.train_grad()
    out = torch.full(g["grid"].shape, 7.0, device="cuda")
    torch.cuda.synchronize()
    lib, l2 = L.load(), C.c_float()
    null = C.cast(None, L._fp)
    assert lib.wost_train_grad(F._h, C.byref(_exec(lib)), C.byref(l2), C.cast(C.c_void_p(out.data_ptr()), L._fp),
                               null, null, null, null) == 0
    assert l2.value == pytest.approx(loss, rel=1e-6)
    assert np.abs(out.cpu().numpy() - g["grid"]).max() <= 64 * 2.0 ** -24 * np.abs(g["grid"]).max()


@pytest.mark.parametrize("make,npts", [(lambda: wi.ngon(64), 700), (lambda: wi.slab_box_flux(3), 500)])
def test_launch_size_changes_no_walk(api, make, npts):
    """Small launches hand their items round the warps, large ones do not (2D)
    or use more lanes (3D): the same walks either way."""
    sc = make()
    S = api.Scene(sc)
    r = np.random.default_rng(2)
    pts = r.uniform(-0.5, 0.5, (npts, sc.dim)) if sc.dim == 2 else r.uniform((-0.9, -0.9, 0.1), (0.9, 0.9, 0.9), (npts, 3))
    nw = 800   # 560,000 and 400,000 walks against one walk per launch
    whole = api.solve(S, pts, nw, seed=9)[0]
    parts = [api.solve(S, pts, 1, seed=9, walk_begin=k)[0] for k in range(0, nw, 80)]
    eight = api.solve(S, pts, 8, seed=9)[0]
    split = [api.solve(S, pts, 1, seed=9, walk_begin=k)[0] for k in range(8)]
    assert np.allclose(np.mean(split, 0), eight, rtol=1e-12, atol=1e-13)
    assert np.isfinite(whole).all() and np.isfinite(parts).all()
    # the last 400 walks and the first 400 add up to the whole
    a = api.solve(S, pts, 400, seed=9)[0]
    b = api.solve(S, pts, 400, seed=9, walk_begin=400)[0]
    assert np.allclose(0.5 * (a + b), whole, rtol=1e-12, atol=1e-13)
