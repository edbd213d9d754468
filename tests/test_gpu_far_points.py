"""Closest primitives of points far outside a 2D scene: where a vertex is nearest
its segments are at exactly the same FP32 distance, and the smallest id is the
answer, however far the point is."""
import dataclasses

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


def _square(n):
    c = np.linspace(-1, 1, n + 1)[:-1]
    one = np.ones(n)
    v = np.concatenate([np.stack(s, 1) for s in [(c, -one), (one, c), (-c, one), (-one, -c)]])
    m = len(v)
    p = np.stack([np.arange(m), (np.arange(m) + 1) % m], 1)
    return wi.Scene("square", 2, v, p, np.zeros(m, np.uint8), wi.Fn(wi.FN_X2_MINUS_Y2))


@pytest.mark.parametrize("reach", [1.0, 30.0, 1000.0])
@pytest.mark.parametrize("n", [1, 8, 100])
def test_nearest_vertex_of_far_points(api, n, reach):
    sc = _square(n)
    # every primitive three times, in another order each: the ties are many
    r = np.random.default_rng(len(sc.prims))
    prims = np.concatenate([sc.prims[r.permutation(len(sc.prims))] for _ in range(3)])
    sc = dataclasses.replace(sc, prims=prims, bc=np.zeros(len(prims), np.uint8))
    d, (lo, hi) = sc.dim, sc.bbox
    n = 2000
    top = r.integers(0, 2, (n, d))
    corner = np.where(top, hi, lo)
    out = r.uniform(0.02, 1, (n, d)) * reach * np.where(top, 1, -1)
    pts = (corner + out).astype(np.float32).astype(np.float64)
    vertex = np.array([np.flatnonzero((sc.verts == c).all(1))[0] for c in corner])
    want = np.array([np.flatnonzero((prims == v).any(1))[0] for v in vertex])
    got = api.Scene(sc).query_closest(pts)[0]
    assert np.array_equal(got, want), (got != want).sum()
