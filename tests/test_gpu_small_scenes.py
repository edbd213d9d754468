"""Scenes whose trees are a single leaf or barely more: which points are inside,
and which of several primitives at the same distance is the closest."""
import dataclasses

import numpy as np
import pytest

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


SCENES = {
    "ngon3": lambda: wi.ngon(3),
    "ngon5": lambda: wi.ngon(5),
    "ngon8": lambda: wi.ngon(8),
    "ngon9": lambda: wi.ngon(9),
    "ngon17": lambda: wi.ngon(17),
    "half_disk": lambda: wi.half_disk(6, 3),
    "star12": lambda: wi.star_polyline(12, seed=3, neumann_frac=0.5),
    "slab1": lambda: wi.slab_box(1),
    "ico0": lambda: wi.displaced_icosphere(subdiv=0, seed=9, neumann_frac=0.5, with_source=False),
}


@pytest.mark.parametrize("name", SCENES)
def test_inside_and_outside(api, name):
    sc = SCENES[name]()
    lo, hi = sc.padded_bbox()
    pts = np.random.default_rng(7).uniform(lo, hi, (3000, sc.dim)).astype(np.float32).astype(np.float64)
    d = oracle.Scene(sc).closest_dirichlet(pts)[1]
    pts = pts[d > 1e-2]   # (an outside point near the boundary is no inside point either, but for rounding)
    # winding number (2D) / solid angle (3D) of the boundary around each point
    V = sc.verts[sc.prims] - pts[:, None, None, :]
    if sc.dim == 2:
        a, b = V[:, :, 0], V[:, :, 1]
        turn = np.arctan2(a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0], (a * b).sum(-1)).sum(1) / (2 * np.pi)
    else:
        a, b, c = V[:, :, 0], V[:, :, 1], V[:, :, 2]
        na, nb, nc = (np.linalg.norm(x, axis=-1) for x in (a, b, c))
        num = (a * np.cross(b, c)).sum(-1)
        den = na * nb * nc + (a * b).sum(-1) * nc + (b * c).sum(-1) * na + (c * a).sum(-1) * nb
        turn = 2 * np.arctan2(num, den).sum(1) / (4 * np.pi)
    inside = np.abs(turn) > 0.5
    assert inside.any() and not inside.all()
    mean = api.solve(api.Scene(sc), pts, 1, maxsteps=8)[0]
    assert np.array_equal(~np.isnan(mean), inside)


@pytest.mark.parametrize("reach", [1.0, 30.0, 1000.0])
def test_ties_in_a_scene_of_one_leaf(api, reach):
    """14 triangles, all tested together: a point whose nearest point is a vertex
    is as far from all triangles there, and takes the smallest id."""
    sc = wi.slab_box(1)
    r = np.random.default_rng(5)
    prims = np.concatenate([sc.prims[r.permutation(12)], sc.prims[:2]])
    sc = dataclasses.replace(sc, prims=prims, bc=np.zeros(14, np.uint8))
    lo, hi = sc.bbox
    top = r.integers(0, 2, (2000, 3))
    corner = np.where(top, hi, lo)
    pts = (corner + r.uniform(0.02, 1, (2000, 3)) * reach * np.where(top, 1, -1)).astype(np.float32).astype(np.float64)
    vertex = [np.flatnonzero((sc.verts == c).all(1))[0] for c in corner]
    want = np.array([np.flatnonzero((prims == v).any(1))[0] for v in vertex])
    got = api.Scene(sc).query_closest(pts)[0]
    assert np.array_equal(got, want), (got != want).sum()
