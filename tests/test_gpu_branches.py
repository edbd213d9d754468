"""Branches of the launches and searches that ordinary scenes do not reach,
each against the general path or the oracle."""
import ctypes as C

import numpy as np
import pytest

import geom_ties as gt
import oracle
import wost_inputs as wi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2410_18944_gb300 import api as A
    return A


def _cone(rings, ratio, sides):
    """A cone of rings that shrink geometrically towards its tip: the trees are
    deep for their size, so the cap tree takes fewer children per node and
    the nearest-first search has little of its stack to choose from."""
    th = 2 * np.pi * np.arange(sides) / sides
    v = np.concatenate([np.stack([0.3 * z * np.cos(th), 0.3 * z * np.sin(th), 0 * th + z], 1)
                        for z in ratio ** np.arange(rings)])
    t = []
    for k in range(rings - 1):
        for i in range(sides):
            a, b = k * sides + i, k * sides + (i + 1) % sides
            t += [(a, b, a + sides), (b, b + sides, a + sides)]
    return wi.Scene("cone", 3, v.astype(np.float32).astype(np.float64), np.array(t), np.zeros(len(t), np.uint8),
                    wi.Fn(wi.FN_X2_MINUS_Y2))


# children per cap node after the stack's limit: 8, 4 (stack almost full), 2
@pytest.mark.parametrize("rings,ratio,sides", [(40, 0.5, 8), (60, 0.7, 8), (60, 0.65, 9), (50, 0.5, 10)])
def test_closest_point_in_deep_trees(api, rings, ratio, sides):
    sc = _cone(rings, ratio, sides)
    r = np.random.default_rng(rings)
    z = np.exp(r.uniform(np.log(1e-4), np.log(1.2), 400))
    off = z[:, None] * r.normal(size=(400, 3)) * r.choice([0.0, 1e-3, 0.1, 0.5], 400)[:, None]
    pts = (np.stack([0 * z, 0 * z, z], 1) + off).astype(np.float32).astype(np.float64)
    O = oracle.Scene(sc)
    d = O.closest_dirichlet(pts)[1]
    g = api.Scene(sc).query_closest(pts)[1]
    assert (np.abs(g - d) <= gt.tie_band(d, O.scale)).all(), np.abs(g - d).max()


def test_lanes_of_a_3d_launch_change_no_walk(api):
    """3D launches above two walks per lane of the GPU use all lanes of a warp,
    smaller ones half of them: the same walks."""
    sc = wi.displaced_icosphere(subdiv=2, seed=9, neumann_frac=0.4, with_source=True)
    S = api.Scene(sc)
    v = np.random.default_rng(2).normal(size=(500, 3))
    pts = 0.6 * v / np.linalg.norm(v, axis=1, keepdims=True)
    whole = api.solve(S, pts, 800, seed=9)[0]    # 400,000 walks
    a = api.solve(S, pts, 400, seed=9)[0]        # 200,000
    b = api.solve(S, pts, 400, seed=9, walk_begin=400)[0]
    assert np.isfinite(whole).all()
    assert np.allclose(0.5 * (a + b), whole, rtol=1e-12, atol=1e-13)


def test_static_solve_in_3d(api):
    import torch

    from paper_2410_18944_gb300 import _lib as L
    for sc in (wi.slab_box_flux(3), wi.displaced_icosphere(subdiv=2, seed=9, neumann_frac=0.4, with_source=True)):
        S = api.Scene(sc)
        lo, hi = sc.padded_bbox()
        pd = torch.tensor(np.random.default_rng(3).uniform(lo, hi, (701, 3)), device="cuda")
        mean, var = (torch.empty(len(pd), dtype=torch.float64, device="cuda") for _ in range(2))
        for nwalks, seed in ((64, 5), (3, 11)):
            steps = C.c_int64()
            L.check(L.load().wost_solve_plain_static(S._h, C.c_void_p(pd.data_ptr()), len(pd), nwalks, 1e-3, 128, seed, None,
                                                     C.c_void_p(mean.data_ptr()), C.c_void_p(var.data_ptr()), C.byref(steps)))
            m, v, st = api.solve(S, pd, nwalks, eps=1e-3, maxsteps=128, seed=seed)
            # the same walks; FP64 atomic sums in another order
            assert steps.value == st["walk_steps"] > 0
            assert torch.allclose(mean, m, rtol=1e-9, atol=1e-12, equal_nan=True)
            assert torch.allclose(var, v, rtol=1e-6, atol=1e-12, equal_nan=True)


def test_3d_batch_with_flux(api):
    """Neumann samples of walks whose scenes differ within a warp."""
    import torch
    jobs = []
    for k, sc in enumerate([wi.slab_box_flux(3), wi.slab_box_flux(1), wi.slab_box(4), wi.slab_box_flux(5)]):
        pts = np.random.default_rng(k).uniform((-0.9, -0.9, 0.1), (0.9, 0.9, 0.9), (11 + 40 * k, 3))
        jobs.append(dict(scene=api.Scene(sc), points=torch.tensor(pts, device="cuda"), nwalks=9, seed=3 + k))
    plan = api.Batch(jobs)
    st = plan.run()
    steps = 0
    for job, mean, var in zip(jobs, plan.mean, plan.var):
        m, v, one = api.solve(job["scene"], job["points"], 9, seed=job["seed"])
        steps += one["walk_steps"]
        assert torch.allclose(mean, m, rtol=1e-9, atol=1e-12)
        assert torch.allclose(var, v, rtol=1e-6, atol=1e-12)
    assert st["walk_steps"] == steps


@pytest.mark.parametrize("K", [8, 16])
def test_decode_in_several_passes(api, K):
    """More positions than two tiles per CTA of the GPU hold: a CTA's tile is
    staging buffer and operand in turn."""
    import torch
    lo, hi = [-1.1] * 3, [1.1] * 3
    F = api.Field(3, lo, hi, K=K, log2_table=12)
    p = wi.random_field_params(3, 3, lo, hi, K=K, log2T=12, grid_scale=0.3)
    F.set_params(**{k: p[k] for k in ("grid", "W1", "W2", "W3", "b3")})
    n = 2 * 2 * torch.cuda.get_device_properties(0).multi_processor_count * 256 + 333
    x = torch.tensor(np.random.default_rng(1).uniform(-1, 1, (n, 3)), device="cuda")
    parts = torch.cat([F.decode(c) for c in x.split(25 * 256)])
    assert torch.equal(F.decode(x), parts)


def test_loss_on_a_side_stream(api):
    import torch

    from paper_2410_18944_gb300.autograd import field_loss
    from test_gpu_streams import field_with_records
    F = field_with_records(api)
    p = wi.random_field_params(3, 3, [-1.1] * 3, [1.1] * 3, K=8, log2T=12, grid_scale=0.3)
    base = [torch.tensor(p[k], dtype=torch.float32, device="cuda") for k in ("grid", "W1", "W2", "W3", "b3")]

    def run():
        # the parameters are computed on the stream that the loss is called on
        torch.cuda._sleep(20_000_000)
        par = [(2 * t).mul(0.5).requires_grad_(True) for t in base]
        loss = field_loss(F, *par)
        loss.backward()
        return loss.detach(), [t.grad for t in par]

    l0, g0 = run()
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        l1, g1 = run()
    torch.cuda.synchronize()
    assert abs(float(l1 - l0)) <= 1e-6 * abs(float(l0))
    for a, b in zip(g1, g0):   # (two orders of FP32 atomic sums)
        assert float((a - b).abs().max()) <= 64 * 2.0 ** -24 * float(b.abs().max())
