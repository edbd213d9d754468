"""Closest-point and silhouette queries where their bounds are sharpest: points
on and just off the boundary (the slab of a patch, the edge-on band), leaf and
node counts around the group sizes, and a scene away from the origin.

Distances are held to the tie band of geom_ties (8 units of 2^-24 of the
distance plus the scene's scale and its distance from the origin); the
silhouette element to its tie rule."""
import dataclasses

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


SCENES = {
    "ngon5": lambda: wi.ngon(5),
    "star17": lambda: wi.star_polyline(17, seed=3, neumann_frac=0.5),
    "star257": lambda: wi.star_polyline(257, seed=8, neumann_frac=0.6),
    "slab1": lambda: wi.slab_box_flux(1),
    "slab4": lambda: wi.slab_box_flux(4),
    "ico0": lambda: wi.displaced_icosphere(subdiv=0, seed=9, neumann_frac=0.5, with_source=False),
    "ico1": lambda: wi.displaced_icosphere(subdiv=1, seed=9, neumann_frac=0.6, with_source=False),
    "ico3": lambda: wi.displaced_icosphere(subdiv=3, seed=4, neumann_frac=0.4, with_source=False),
}


def _points(sc, n, seed):
    """Points at 0, 1e-6, 1e-4, 1e-2 and 0.3 of the scale inside a random
    boundary point (a quarter of them at a vertex), FP32 values."""
    r = np.random.default_rng(seed)
    V, P = sc.verts, sc.prims
    d = V.shape[1]
    t = r.integers(0, len(P), n)
    w = r.dirichlet(np.ones(d), n)
    at_vertex = r.random(n) < 0.25
    w[at_vertex] = np.eye(d)[r.integers(0, d, at_vertex.sum())]
    c = (V[P[t]] * w[:, :, None]).sum(1)
    scale = np.linalg.norm(V.max(0) - V.min(0))
    off = r.choice([0.0, 1e-6, 1e-4, 1e-2, 0.3], n) * scale
    return (c + off[:, None] * gt.inward_normals(sc)[t]).astype(np.float32).astype(np.float64)


@pytest.mark.parametrize("shift", [0.0, 4.0])
@pytest.mark.parametrize("name", SCENES)
def test_queries_near_the_boundary(api, name, shift):
    sc = SCENES[name]()
    # FP32-representable vertices: the queries' own input rounding stays out
    sc = dataclasses.replace(sc, verts=(sc.verts + shift).astype(np.float32).astype(np.float64))
    pts = _points(sc, 256, seed=len(name))
    S, O = api.Scene(sc), oracle.Scene(sc)
    scale = O.scale + abs(shift) * np.sqrt(sc.verts.shape[1])
    gi, gd = S.query_closest(pts)
    od = O.closest_dirichlet(pts)[1]
    band = np.array([gt.tie_band(x, scale) for x in od])
    assert (gi >= 0).all()
    assert (np.abs(gd - od) <= band).all(), np.abs(gd - od).max()
    if shift or not (sc.bc == 1).any():
        return   # the silhouette rule's bands are those of a scene at the origin
    el = gt.silhouette_elements(sc)
    key_index = {int(k): i for i, k in enumerate(el[4])}
    nin = gt.inward_normals(sc)
    gk, gs = S.query_silhouette(pts)
    bad = [i for i in range(len(pts))
           if not gt.silhouette_answer_ok(gk[i], gs[i], key_index,
                                          gt.silhouette_candidates(sc, el, nin, pts[i], scale), scale)]
    assert not bad, [(i, gk[i], gs[i]) for i in bad[:5]]
