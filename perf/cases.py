"""Timed cases of the library: what its users have it do, through the public
binding (``paper_2410_18944_gb300.api`` and ``autograd``), with the outputs of
each pass.

The kinds of work, and what each stands for in real use:

  plain    wost_solve without a field: the reference solve of a study, the
           equal-time comparison, a quick look at a few points.
  guided   wost_solve with a trained field that no longer learns: the walks
           past ``train_until_wpp``, or a field kept from an earlier solve.
  train    wost_solve with online training from a fresh field: one training
           batch of walks and the update of the field.
  decode   wost_field_decode: the mixture parameters at given positions (maps
           of the learned distribution, the network on its own).
  loss     the field's training loss and its gradients, forward and backward,
           as ``torch`` code that optimises the field with its own optimiser
           calls them.
  batch    a plan of many scenes, replayed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import wost_inputs as wi
from paper_2410_18944_gb300 import api, autograd

EPS = 1e-3
LEVELS, FEATURES, BASE_RES = 16, 2, 16
PRIMES = (1, 2654435761, 805459861)


def listed():
    return [
        # the smallest solve: the 64-segment Laplace problem on its 32 x 32 grid
        dict(name="plain_small", kind="plain", scene="ngon", nseg=64, res=32, points=812, walks=64, rr=0),
        # the 2D problem of the benchmark, every point of its grid
        dict(name="plain_star", kind="plain", scene="star", nseg=4096, shape=2, res=512, points=0, walks=8, rr=0),
        # 3D with source terms: the icosphere's slice
        dict(name="plain_icosphere", kind="plain", scene="icosphere", subdiv=6, shape=3, res=256, points=0, walks=8, rr=0),
        # 3D on a mesh of a million triangles, a subset of its slice
        dict(name="plain_genus3", kind="plain", scene="genus3", n=330, res=1024, points=32768, walks=4, rr=0),
        # nonzero Neumann flux, long walks ended by roulette
        dict(name="plain_flux", kind="plain", scene="slab_flux", nquad=16, res=0, points=4093, walks=32, rr=64),
        # walks with a trained field
        dict(name="guided_star", kind="guided", scene="star", nseg=4096, shape=2, res=512, points=0, walks=4, K=8, c_mode=0),
        dict(name="guided_icosphere", kind="guided", scene="icosphere", subdiv=6, shape=3, res=256, points=16001, walks=4,
             K=8, c_mode=0),
        # one training batch: four walks per point of the star's grid; two on the million-triangle mesh
        dict(name="train_star", kind="train", scene="star", nseg=4096, shape=2, res=512, points=0, walks=4, K=8),
        dict(name="train_genus3", kind="train", scene="genus3", n=330, res=1024, points=65536, walks=2, K=8),
        # the network on its own, over a large point set of odd size
        dict(name="decode", kind="decode", dim=3, points=1000003, K=8, grid_type=0),
        # loss and gradients of one minibatch
        dict(name="loss_grad", kind="loss", dim=3, records=262144, K=8),
        # many uneven scenes in one plan
        dict(name="batch", kind="batch", jobs=12, shape=4, seg_lo=256, seg_hi=16384, pts_lo=1024, pts_hi=65536, wpp_lo=4,
             wpp_hi=32, guided=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scene(rng, walks_max):
    """A scene and a point count whose walks stay below walks_max[scene]."""
    scene = rng.choice(["star", "star", "icosphere", "icosphere", "genus3"])
    c = dict(scene=scene)
    if scene == "star":
        c.update(nseg=_log_int(rng, 256, 16384), shape=rng.randint(1, 1 << 20), res=_log_int(rng, 32, 512))
    elif scene == "icosphere":
        c.update(subdiv=rng.choice([4, 5, 6]), shape=rng.randint(1, 1 << 20), res=_log_int(rng, 48, 256))
    else:
        c.update(n=330, res=1024)
    c["points"] = _log_int(rng, 300, 60000)
    c["walks"] = max(1, min(_log_int(rng, 1, 64), walks_max[scene] // c["points"]))
    return c


def draw(rng):
    kind = rng.choice(["plain", "plain", "guided", "guided", "train", "train", "decode", "loss", "batch"])
    if kind == "plain":
        if rng.random() < 0.25:
            return dict(kind=kind, scene=rng.choice(["slab_flux", "half_disk_flux"]), nquad=_log_int(rng, 3, 24),
                        res=0, points=_log_int(rng, 100, 4000), walks=_log_int(rng, 4, 32),
                        rr=rng.choice([0, 32, 64]))
        c = _draw_scene(rng, dict(star=1400000, icosphere=300000, genus3=120000))
        return dict(kind=kind, rr=rng.choice([0, 0, 64]), **c)
    if kind == "guided":
        c = _draw_scene(rng, dict(star=600000, icosphere=120000, genus3=100000))
        return dict(kind=kind, K=rng.choice([8, 8, 4, 16]), c_mode=rng.choice([0, 0, 1]), **c)
    if kind == "train":
        c = _draw_scene(rng, dict(star=600000, icosphere=120000, genus3=100000))
        return dict(kind=kind, K=rng.choice([8, 8, 4, 16]), **c)
    if kind == "decode":
        return dict(kind=kind, dim=rng.choice([2, 3]), points=_log_int(rng, 1000, 3000000),
                    K=rng.choice([8, 8, 4, 16]), grid_type=0)
    if kind == "loss":
        return dict(kind=kind, dim=rng.choice([2, 3]), records=_log_int(rng, 1000, 262144),
                    K=rng.choice([8, 8, 4, 16]))
    lo = _log_int(rng, 256, 4096)
    return dict(kind=kind, jobs=rng.randint(3, 16), shape=rng.randint(1, 1000), seg_lo=256, seg_hi=_log_int(rng, 1024, 16384), pts_lo=lo,
                pts_hi=lo * rng.randint(2, 8), wpp_lo=2, wpp_hi=rng.randint(4, 16), guided=rng.choice([0, 1]))


# ---- inputs ------------------------------------------------------------------

def _stream(seed, what):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, what])


@functools.lru_cache(maxsize=2)
def _genus3(n, res):
    """The genus-3 mesh, its scene handle and its slice's points.  Meshing and
    the scene take much longer than a solve; a program keeps both and solves
    on them again and again."""
    sc, pts = wi.config_genus3(res=res, n=n)
    return api.Scene(sc), pts


def _subset(pts, case, seed):
    n = case.get("points", 0)
    if n <= 0 or n >= len(pts):
        return pts
    return pts[np.sort(_stream(seed, 1).choice(len(pts), n, replace=False))]


def _scene_points(case, seed):
    """(scene handle, query points) of a case; the seed picks the points and
    moves them a little towards the origin, about which the domains with a
    grid of points are star-shaped."""
    kind = case["scene"]
    toward = 1 - 0.01 * _stream(seed, 2).random()
    if kind == "ngon":
        sc = wi.ngon(case["nseg"])
        pts = wi.grid_points_2d(case["res"], (-1, -1), (1, 1))
        return api.Scene(sc), toward * _subset(pts[wi.inside_polygon_mask(sc, pts)], case, seed)
    if kind == "star":
        sc, pts = wi.config_star_guided(res=case["res"], nseg=case["nseg"], seed=case["shape"])
        return api.Scene(sc), toward * _subset(pts, case, seed)
    if kind == "icosphere":
        sc, pts = wi.config_3d_guided(res=case["res"], subdiv=case["subdiv"], seed=case["shape"])
        return api.Scene(sc), toward * _subset(pts, case, seed)
    if kind == "genus3":
        scene, pts = _genus3(case["n"], case["res"])
        return scene, _subset(pts, case, seed)
    r = _stream(seed, 4)
    if kind == "slab_flux":
        sc = wi.slab_box_flux(case["nquad"])
        return api.Scene(sc), r.uniform((-0.95, -0.95, 0.05), (0.95, 0.95, 0.95), (case["points"], 3))
    sc = wi.half_disk_flux(8 * case["nquad"], 4 * case["nquad"], poisson=True)
    rad, th = np.sqrt(r.uniform(0.01, 0.85, case["points"])), r.uniform(0.05, math.pi - 0.05, case["points"])
    return api.Scene(sc), np.stack([rad * np.cos(th), rad * np.sin(th)], 1)


def _cuda(pts):
    return torch.tensor(np.ascontiguousarray(pts), dtype=torch.float64, device="cuda")


def _params(dim, K, seed, lo, hi, grid_type=0):
    """Parameters of a field after training: features and outputs of order one."""
    p = wi.random_field_params(dim, int(_stream(seed, 5).integers(1, 1 << 30)), lo, hi, K=K,
                               log2T=16 if dim == 2 else 19, grid_scale=0.3, grid_type=grid_type)
    return {k: np.ascontiguousarray(p[k], np.float32) for k in ("grid", "W1", "W2", "W3", "b3")}


def _walk_seed(seed):
    return int(_stream(seed, 6).integers(1, 1 << 40))


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("plain", "guided", "train"):
        scene, pts = _scene_points(case, seed)
        s = dict(kind=kind, scene=scene, points=_cuda(pts), walks=case["walks"], seed=_walk_seed(seed))
        if kind == "plain":
            s["exec"] = dict(rr_depth=case["rr"]) if case["rr"] else {}
            s["maxsteps"] = 1024 if case["rr"] else 128
            return s
        lo, hi = scene.bbox()
        s["field"] = api.Field(scene.dim, lo, hi, K=case["K"])
        if kind == "guided":
            s["field"].set_params(**_params(scene.dim, case["K"], seed, lo, hi))
            s["exec"] = dict(c_mode=case["c_mode"], c_fixed=0.5)
        else:
            s["fresh"] = s["field"].get_params()
        return s
    if kind == "decode":
        dim = case["dim"]
        lo, hi = [-1.1] * dim, [1.1] * dim
        field = api.Field(dim, lo, hi, K=case["K"], grid_type=case["grid_type"])
        field.set_params(**_params(dim, case["K"], seed, lo, hi, case["grid_type"]))
        return dict(kind=kind, field=field, points=_cuda(_stream(seed, 7).uniform(-1, 1, (case["points"], dim))))
    if kind == "loss":
        dim = case["dim"]
        lo, hi = [-1.1] * dim, [1.1] * dim
        field = api.Field(dim, lo, hi, K=case["K"])
        field.set_records(_records(dim, case["records"], seed))
        p = _params(dim, case["K"], seed, lo, hi)
        return dict(kind=kind, field=field,
                    params=[torch.tensor(p[k], device="cuda", requires_grad=True) for k in ("grid", "W1", "W2", "W3", "b3")])
    jobs = []
    for j in wi.config_batch(case["jobs"], seed=case["shape"], seg_range=(case["seg_lo"], case["seg_hi"]),
                             points_range=(case["pts_lo"], case["pts_hi"]), wpp_range=(case["wpp_lo"], case["wpp_hi"])):
        scene = api.Scene(j.scene)
        pts = wi.star_interior_points(j.scene, len(j.points), seed=(seed + 7919 * len(jobs)) & 0x7FFFFFFF)
        job = dict(scene=scene, points=_cuda(pts), nwalks=j.nwalks, seed=_walk_seed(seed + len(jobs)))
        if case["guided"]:
            lo, hi = scene.bbox()
            job["field"] = api.Field(2, lo, hi)
            job["field"].set_params(**_params(2, 8, seed + len(jobs), lo, hi))
        jobs.append(job)
    return dict(kind=kind, plan=api.Batch(jobs, guided=bool(case["guided"])))


def _records(dim, n, seed):
    """Training records as walks leave them: positions in the domain, about a
    third of them on the Neumann boundary with directions on its inner side,
    densities of the sampled mixture, heavy-tailed targets with some zeros."""
    r = _stream(seed, 9)
    rec = np.zeros((n, 12), np.float32)
    rec[:, :dim] = r.uniform(-1, 1, (n, dim))
    nu = r.normal(size=(n, dim))
    nu /= np.linalg.norm(nu, axis=1, keepdims=True)
    nrm = r.normal(size=(n, dim))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    on = r.random(n) < 0.3
    side = np.sign((nu * nrm).sum(1))
    nu[on] *= np.where(side[on] == 0, 1, side[on])[:, None]
    rec[:, 3:3 + dim] = nu
    rec[on, 6:6 + dim] = nrm[on]
    rec[on, 9] = 1
    rec[:, 10] = r.uniform(0.03, 0.4, n)
    rec[:, 11] = np.where(r.random(n) < 0.05, 0.0, 0.4 * np.exp(0.5 * r.normal(size=n)))
    return rec


# ---- one pass ------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "plain":
        mean, var, _ = api.solve(state["scene"], state["points"], state["walks"], eps=EPS, maxsteps=state["maxsteps"],
                                 seed=state["seed"], **state["exec"])
        return {"mean": mean, "var": var}
    if kind == "guided":
        mean, var, _ = api.solve(state["scene"], state["points"], state["walks"], eps=EPS, guided=True,
                                 field=state["field"], seed=state["seed"], **state["exec"])
        return {"mean": mean, "var": var}
    if kind == "train":
        field = state["field"]
        field.set_params(**state["fresh"])   # a new problem starts from a fresh field
        mean, var, _ = api.solve(state["scene"], state["points"], state["walks"], eps=EPS, guided=True, field=field,
                                 train=1, batch_wpp=state["walks"], seed=state["seed"])
        return {"mean": mean, "var": var, "field": field.get_params()}
    if kind == "decode":
        return {"raw": state["field"].decode(state["points"])}
    if kind == "loss":
        for p in state["params"]:
            p.grad = None
        loss = autograd.field_loss(state["field"], *state["params"])
        loss.backward()
        return {"loss": loss.detach(), "grads": [p.grad for p in state["params"]]}
    state["plan"].run()
    return {"mean": state["plan"].mean, "var": state["plan"].var}


# ---- what a pass cannot do without -----------------------------------------------

def _mlp_flops(dim, K):
    return 2.0 * (32 * 64 + 64 * 64 + 64 * ((dim + 2) * K + 1))


def _corner_bytes(dim):
    return LEVELS * 2.0 ** dim * FEATURES * 2


def _field_floats(dim, K):
    nout = (dim + 2) * K + 1
    return LEVELS * (1 << (16 if dim == 2 else 19)) * FEATURES + 64 * 32 + 64 * 64 + 65 * nout


def _scene_bytes(case):
    """The boundary, read once: vertices of the primitives in FP32."""
    k = case["scene"]
    if k in ("star", "ngon"):
        return 16.0 * case["nseg"]
    if k == "icosphere":
        return 36.0 * 20 * 4 ** case["subdiv"]
    if k == "genus3":
        return 36.0 * 9.1 * case["n"] ** 2
    return 36.0 * 12 * case["nquad"] ** 2 if k == "slab_flux" else 16.0 * 12 * case["nquad"]


def _points(case):
    if case["points"]:
        return case["points"]
    return {"star": 0.66, "icosphere": 0.72, "genus3": 0.49}[case["scene"]] * case["res"] ** 2


def work(case):
    kind = case["kind"]
    if kind in ("plain", "guided", "train"):
        dim = 2 if case["scene"] in ("ngon", "star", "half_disk_flux") else 3
        n = _points(case)
        walks = n * case["walks"]
        # a walk is about 20 (2D) or 32 (3D) steps; a step cannot do without
        # one closest-point test, one silhouette test and one ray test
        steps = walks * (20 if dim == 2 else 32)
        b = _scene_bytes(case) + n * 8.0 * (dim + 2)
        f = steps * (60.0 if dim == 2 else 200.0)
        if kind != "plain":
            b += 4.0 * _field_floats(dim, case["K"])
            f += steps * _mlp_flops(dim, case["K"])
        if kind == "train":
            # each step leaves a record that is read back once; the update
            # reads and writes the parameters and both moments
            b += steps * 96.0 + 24.0 * _field_floats(dim, case["K"])
            f += steps * 3 * _mlp_flops(dim, case["K"])
        return {"bytes": b, "flops": f}
    if kind == "decode":
        d, n = case["dim"], case["points"]
        nout = (d + 2) * case["K"] + 1
        grid = LEVELS * (1 << (16 if d == 2 else 19)) * FEATURES * 2.0
        return {"bytes": n * (8.0 * d + 4.0 * nout) + min(grid, n * _corner_bytes(d)), "flops": n * _mlp_flops(d, case["K"])}
    if kind == "loss":
        d, n = case["dim"], case["records"]
        return {"bytes": n * 48.0 + 8.0 * _field_floats(d, case["K"]), "flops": 4.0 * n * _mlp_flops(d, case["K"])}
    pts = case["jobs"] * math.sqrt(case["pts_lo"] * case["pts_hi"])
    steps = 20.0 * pts * math.sqrt(case["wpp_lo"] * case["wpp_hi"])
    return {"bytes": pts * 32.0 + case["jobs"] * 16.0 * math.sqrt(case["seg_lo"] * case["seg_hi"]),
            "flops": steps * (60.0 + (_mlp_flops(2, 8) if case["guided"] else 0))}


# ---- the same in 64 bits -----------------------------------------------------------

def exact(case, seed):
    """Network outputs, and the training loss with its gradients, in 64 bits.
    The solves are Monte Carlo estimates on the library's own random streams:
    there is no value of theirs to give."""
    kind = case["kind"]
    if kind not in ("decode", "loss"):
        return None
    dim, K = case["dim"], case["K"]
    lo, hi = [-1.1] * dim, [1.1] * dim
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    p = _params(dim, K, seed, lo, hi, case.get("grid_type", 0))
    par = [torch.tensor(p[k], dtype=torch.float64, device=dev) for k in ("grid", "W1", "W2", "W3", "b3")]
    if kind == "decode":
        x = torch.tensor(_stream(seed, 7).uniform(-1, 1, (case["points"], dim)), device=dev)
        return {"raw": torch.cat([_network64(par, c, dim, lo, hi) for c in x.split(1 << 17)])}
    par = [t.requires_grad_(True) for t in par]
    rec = torch.tensor(_records(dim, case["records"], seed), dtype=torch.float64, device=dev)
    loss = sum(_loss64(par, r, dim, K, lo, hi) for r in rec.split(1 << 16)) / len(rec)
    loss.backward()
    return {"loss": loss.detach(), "grads": [t.grad for t in par]}


def _network64(par, x, dim, lo, hi):
    grid, W1, W2, W3, b3 = par
    T = grid.shape[1]
    lo_t, hi_t = torch.tensor(lo, dtype=x.dtype, device=x.device), torch.tensor(hi, dtype=x.dtype, device=x.device)
    u = (x - lo_t) / (hi_t - lo_t)
    feats = []
    for l, N in enumerate(wi.level_resolutions(LEVELS, BASE_RES, 2048 if dim == 2 else 512)):
        q = u * N
        cell = q.floor().clamp(0, N - 1)
        fr, cell = q - cell, cell.long()
        acc = 0
        for m in range(1 << dim):
            w, idx, side = 1.0, 0, 1
            for k in range(dim):
                bit = (m >> k) & 1
                w = w * (fr[:, k] if bit else 1 - fr[:, k])
                v = cell[:, k] + bit
                if (N + 1) ** dim <= T:
                    idx, side = idx + side * v, side * (N + 1)
                else:
                    idx = idx ^ ((v * PRIMES[k]) & 0xFFFFFFFF)
            acc = acc + w[:, None] * grid[l][idx & (T - 1) if (N + 1) ** dim > T else idx]
        feats.append(acc)
    h = torch.cat(feats, 1)
    return torch.relu(torch.relu(h @ W1.T) @ W2.T) @ W3.T + b3


def _loss64(par, rec, dim, K, lo, hi, e_sel=0.2):
    """Sum of -(p_t / q) [log p_g + e log(c p_g0 + (1 - c) p_u)], p_g0 held fixed."""
    raw = _network64(par, rec[:, :dim], dim, lo, hi)
    mu = raw[:, :K * dim].reshape(-1, K, dim)
    mu = mu / mu.norm(dim=2, keepdim=True)
    kap = raw[:, K * dim:K * dim + K].clamp(-8, 8).exp()
    lam = torch.softmax(raw[:, K * dim + K:K * dim + 2 * K], 1)
    c = torch.sigmoid(raw[:, -1])
    nu, nrm, on = rec[:, 3:3 + dim], rec[:, 6:6 + dim], rec[:, 9] != 0
    norm = 1 / (2 * math.pi * torch.special.i0e(kap)) if dim == 2 else kap / (2 * math.pi * -torch.expm1(-2 * kap))
    refl = nu - 2 * (nu * nrm).sum(1, keepdim=True) * nrm
    val = (kap * ((mu * nu[:, None]).sum(2) - 1)).exp()
    val = val + on[:, None] * (kap * ((mu * refl[:, None]).sum(2) - 1)).exp()
    pg = (lam * norm * val).sum(1)
    pu = torch.where(on, 2.0, 1.0) / (2 * math.pi if dim == 2 else 4 * math.pi)
    keep = (rec[:, 11] > 0) & (rec[:, 10] > 0)
    w = torch.where(keep, rec[:, 11] / rec[:, 10], 0.0)
    return -(w * (pg.log() + e_sel * (c * pg.detach() + (1 - c) * pu).log())).sum()
