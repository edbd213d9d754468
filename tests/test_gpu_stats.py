"""The launch statistics' algorithmic bytes: scenes whose three trees are one
node each, so that every query visits exactly one node."""
import numpy as np
import pytest

import wost_inputs as wi

pytestmark = pytest.mark.gpu

# bytes of a visited node (closest point: caps; silhouette: boxes and facing
# bounds; rays: boxes), a segment or triangle, a silhouette element
BYTES = {2: dict(caps=64, sil=96, box=48, prim=16, elem=32), 3: dict(caps=512, sil=224, box=128, prim=48, elem=48)}


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2410_18944_gb300 import api as A
    return A


def _expected(dim, st, neumann, guided):
    b = BYTES[dim]
    going = st["walk_steps"] - st["walks"]   # every walk ends in one terminal step
    queries = st["walk_steps"] + (2 * going if neumann else 0)
    again = st["node_visits"] - queries      # closest points searched a second time, in the boxes (3D)
    assert again >= 0 if dim == 3 else again == 0
    nodes = b["caps"] * st["walk_steps"] + b["box"] * again + ((b["sil"] + b["box"]) * going if neumann else 0)
    prims = b["prim"] * (st["dir_prim_visits"] + st["neu_prim_visits"]) + b["elem"] * st["sil_prim_visits"]
    corners = 64 * 2 ** dim * going if guided else 0
    return nodes + prims + corners + st["walks"] * (8 * dim + 16)


@pytest.mark.parametrize("kind", ["solve", "guided", "batch"])
@pytest.mark.parametrize("make,neumann", [(lambda: wi.ngon(8), False), (lambda: wi.half_disk(6, 3), True),
                                          (lambda: wi.slab_box(1), True)], ids=["ngon", "half_disk", "slab"])
def test_bytes_of_visited_nodes(api, make, neumann, kind):
    import torch
    sc = make()
    r = np.random.default_rng(1)
    lo, hi = ((-0.5, 0.1), (0.5, 0.5)) if sc.dim == 2 else ((-0.8, -0.8, 0.1), (0.8, 0.8, 0.9))
    pts = torch.tensor(r.uniform(lo, hi, (300, sc.dim)), device="cuda")
    S = api.Scene(sc)
    if kind == "batch":
        st = api.Batch([dict(scene=S, points=pts, nwalks=8, seed=5)]).run()
    elif kind == "solve":
        st = api.solve(S, pts, 8, seed=5)[2]
    else:
        st = api.solve(S, pts, 8, seed=5, guided=True, field=api.Field(sc.dim, *S.bbox()))[2]
    assert st["walks"] == 8 * len(pts)
    assert st["alg_bytes"] == _expected(sc.dim, st, neumann, kind == "guided")
