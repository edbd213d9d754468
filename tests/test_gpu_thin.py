"""Closest points of thin boundaries (slits, fins): a patch much longer than it
is thick, at random rotations, queried where it and the walls around it are
about as far.  Distances are held to the tie band of geom_ties."""
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


def _square_with_slit(n, thick, angle):
    """[-1, 1]^2 with 8 segments a side around a wedge of length 1 and half
    thickness `thick` at its blunt end, n segments a long side; and its
    directions (along, across)."""
    c = np.linspace(-1, 1, 9)[:-1]
    one = np.ones(8)
    outer = np.concatenate([np.stack(s, 1) for s in [(c, -one), (one, c), (-c, one), (-one, -c)]])
    x = np.linspace(-0.5, 0.5, n + 1)
    y = thick * (0.5 - x)
    hole = np.concatenate([np.stack([x, y], 1), np.stack([x, -y], 1)[-2::-1]])   # clockwise
    rot = np.array([[np.cos(angle), -np.sin(angle)], [np.sin(angle), np.cos(angle)]])
    loop = lambda k, m: np.stack([k + np.arange(m), k + (np.arange(m) + 1) % m], 1)
    v = np.concatenate([outer, hole @ rot.T]).astype(np.float32).astype(np.float64)
    prims = np.concatenate([loop(0, len(outer)), loop(len(outer), len(hole))])
    return wi.Scene("slit", 2, v, prims, np.zeros(len(prims), np.uint8), wi.Fn(wi.FN_X2_MINUS_Y2)), rot


def _box_with_needle(n, thick, angle):
    """[-1, 1]^3 around a three-sided needle of length 1 and radius `thick` at
    its blunt end, its sides cut into n strips; and its directions (along,
    across, across)."""
    box = wi.slab_box(4)
    walls = box.verts * (1, 1, 2) - (0, 0, 1)
    rot = np.linalg.qr(np.random.default_rng(int(1000 * angle)).normal(size=(3, 3)))[0]
    rot[:, 2] *= np.sign(np.linalg.det(rot))
    th = 2 * np.pi / 3 * np.arange(3)
    v = [np.stack([0 * th + h, thick * (0.5 - h) * np.cos(th), thick * (0.5 - h) * np.sin(th)], 1)
         for h in np.linspace(-0.5, 0.5, n + 1)[:-1]]
    v = np.concatenate(v + [np.array([[0.5, 0, 0]])])
    t = [(0, 1, 2)]   # normals into the needle: out of the domain
    for k in range(n):
        for i in range(3):
            a, b = 3 * k + i, 3 * k + (i + 1) % 3
            t += [(a, 3 * n, b)] if k == n - 1 else [(a, a + 3, b), (b, a + 3, b + 3)]
    verts = np.concatenate([walls, v @ rot.T]).astype(np.float32).astype(np.float64)
    prims = np.concatenate([box.prims, np.array(t) + len(walls)])
    return wi.Scene("needle", 3, verts, prims, np.zeros(len(prims), np.uint8), wi.Fn(wi.FN_X2_MINUS_Y2)), rot


@pytest.mark.parametrize("thick", [2e-4, 2e-5])
@pytest.mark.parametrize("n", [1, 2, 8])
@pytest.mark.parametrize("make", [_square_with_slit, _box_with_needle])
def test_closest_point_of_a_thin_patch(api, make, n, thick):
    for angle in (0.3, 0.7, 1.1, 1.9, 2.6):
        sc, rot = make(n, thick, angle)
        along, across = rot[:, 0], rot[:, 1]
        lo, hi = sc.bbox
        r = np.random.default_rng(int(100 * angle) + n)
        p0 = r.uniform(-0.5, 0.5, 500)[:, None] * along
        # on lines that leave the patch sideways: where the walls are as far
        a, b = np.zeros(len(p0)), np.full(len(p0), 2.0)
        for _ in range(50):
            t = 0.5 * (a + b)
            x = p0 + t[:, None] * across
            nearer = t - thick < np.minimum(x - lo, hi - x).min(1)
            a, b = np.where(nearer, t, a), np.where(nearer, b, t)
        t = a + r.uniform(-1.0, 0.0, len(a)) * thick
        pts = (p0 + t[:, None] * across).astype(np.float32).astype(np.float64)
        O = oracle.Scene(sc)
        d = O.closest_dirichlet(pts)[1]
        err = np.abs(api.Scene(sc).query_closest(pts)[1] - d)
        assert (err <= gt.tie_band(d, O.scale)).all(), (angle, err.max())
