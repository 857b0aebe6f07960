"""The work a user of the library has it do, as cases that can be timed and checked.

A case is a dict of plain values.  ``listed()`` gives the fixed ones, ``draw(rng)``
one more of the same ranges, ``prepare(case, seed)`` what a program has in hand
before the call (clouds, bands with mid-fit values, records, meshes), ``run(state)``
one pass through the public entry points, ``work(case)`` the bytes and operations
the path cannot do without, and ``exact(case, seed)`` the results in 64 bits where
plain torch gives them in a few seconds.

Clouds are noisy samples of the surfaces the benchmark names (sphere, union of
ellipsoids and a torus, superquadrics, furnished room, mixed unions); grid values
are the surface's approximate signed distance plus a tenth of a cell of noise, and
the Adam moments are non-zero, as in the middle of a fit."""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2308_13175_gb300 import binding as gb
from paper_2308_13175_gb300 import metrics
from paper_2308_13175_gb300.autograd import gridpull_loss
from paper_2308_13175_gb300.fit import FitStep

WEIGHTS = (1.0, 1.0, 0.005)
LR = 1e-3
STEP0 = 100  # fitting steps before the measured one (the moments are then in use)


def listed():
    return [
        # The smallest fit: 5,000 points on a sphere, dense 64^3 grid, all 50,000 queries in each step.
        # Calls this small are launches and latency.
        {"name": "sphere_fit", "kind": "fit", "cloud": "sphere", "shape": 0, "points": 5_000, "R": 64, "M1": -1,
         "M2": -1, "B": 50_000, "steps": 1, "deterministic": False},
        # The paper's own settings, the defaults of fit_cloud: 256^3, M1 = 3, M2 = 14, 50,000 queries a step.
        {"name": "shape_fit", "kind": "fit", "cloud": "object", "shape": 2, "points": 30_000, "R": 256, "M1": 3,
         "M2": 14, "B": 50_000, "steps": 1, "deterministic": False},
        # A single scanned object at the benchmark's size.
        {"name": "object_fit", "kind": "fit", "cloud": "object", "shape": 1, "points": 100_000, "R": 256, "M1": 2,
         "M2": 2, "B": 262_144, "steps": 1, "deterministic": False},
        # The largest: an indoor scene of 10 M points on a 1024^3 band, two pipelined steps.
        {"name": "scene_fit", "kind": "fit", "cloud": "room", "shape": 2, "points": 10_000_000, "R": 1024, "M1": 2,
         "M2": 2, "B": 2_097_152, "steps": 2, "deterministic": False},
        # Many clouds of uneven size fitted together, one launch a stage.
        {"name": "collection_fit", "kind": "multi", "clouds": 20, "shape": 3, "j_min": 5_000, "j_max": 500_000,
         "deterministic": False},
        # Nearest points of a large batch whose source points are known (the search a fitting step makes).
        {"name": "superquadric_nn", "kind": "nn", "cloud": "superquadric", "shape": 4, "points": 2_000_000, "R": 512,
         "queries": 1_500_001, "seeded": True},
        # Loss and gradient of a caller's own records in no spatial order, no count handed over (a custom loop).
        {"name": "object_step", "kind": "step", "cloud": "object", "shape": 1, "points": 100_000, "R": 256, "M1": 3,
         "M2": 14, "B": 262_144, "deterministic": False},
        # Bitwise repeatable step and update on a large object.
        {"name": "superquadric_det", "kind": "step", "cloud": "superquadric", "shape": 4, "points": 2_000_000,
         "R": 512, "M1": 2, "M2": 2, "B": 4_194_304, "deterministic": True},
        # The loss as a torch.autograd.Function, forward and backward.
        {"name": "object_autograd", "kind": "autograd", "cloud": "object", "shape": 1, "points": 100_000, "R": 256,
         "M1": 2, "M2": 2, "B": 262_144},
        # The allocation-free form on a dense grid of the caller's, a ragged batch.
        {"name": "dense_noalloc", "kind": "dense", "shape": 0, "R": 128, "B": 99_999},
        # The band of a new cloud, with the sampling widths (every fit begins with it).
        {"name": "object_build", "kind": "build", "cloud": "object", "shape": 1, "points": 100_000, "R": 256, "M1": 2,
         "M2": 2, "knn": 50},
        # The end of a reconstruction: the mesh of the fitted field, scored against oriented reference points.
        {"name": "object_mesh", "kind": "mesh", "cloud": "object", "shape": 1, "points": 100_000, "R": 256, "M1": 2,
         "M2": 2, "reference": 100_000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _resolution(rng, points, top):
    """A power of two near the grid whose cells hold a few points each."""
    r = 2 ** round(math.log2(math.sqrt(points) * rng.uniform(0.6, 1.7)))
    return max(64, min(top, r))


def draw(rng):
    kind = rng.choice(["fit", "fit", "multi", "nn", "step", "autograd", "dense", "build", "mesh"])
    if kind == "multi":
        j_min = _log(rng, 2_000, 20_000)
        return {"kind": kind, "clouds": rng.randint(2, 20), "shape": rng.randrange(1000), "j_min": j_min,
                "j_max": j_min * rng.randint(2, 25), "deterministic": rng.random() < 0.3}
    if kind == "dense":
        return {"kind": kind, "shape": rng.randrange(1000), "R": 2 ** rng.randint(4, 8), "B": _log(rng, 500, 1_000_000)}
    cloud = rng.choice(["sphere", "object", "superquadric", "room"])
    case = {"kind": kind, "cloud": cloud, "shape": rng.randrange(1000), "points": _log(rng, 2_000, 2_000_000)}
    if kind in ("build", "mesh"):
        case["points"] = _log(rng, 2_000, 500_000)
    case["R"] = _resolution(rng, case["points"], 256 if kind in ("build", "mesh") else 512)
    if kind == "nn":
        seeded = rng.random() < 0.7
        return {**case, "queries": _log(rng, 1_000, 3_000_000 if seeded else 300_000), "seeded": seeded}
    wide = case["R"] <= 256 and rng.random() < 0.4
    case["M1"], case["M2"] = (3, 14) if wide else (-1, -1) if case["R"] == 64 and rng.random() < 0.4 else (2, 2)
    if kind == "build":
        return {**case, "knn": rng.choice([10, 20, 50])}
    if kind == "mesh":
        return {**case, "reference": _log(rng, 2_000, 200_000)}
    case["B"] = _log(rng, max(500, case["points"] // 8), min(4_000_000, 10 * case["points"]))
    if kind == "fit":
        case["steps"] = rng.choice([1, 1, 2])
    if kind in ("fit", "step"):
        case["deterministic"] = rng.random() < 0.4
    return case


# ------------------------------------------------------------------ surfaces
class Shape:
    """A union of primitives (kind, centre, rotation local -> world, parameters); for a room the first box is the
    shell, seen from inside."""

    def __init__(self, cloud: str, shape: int):
        r = random.Random("%s %d" % (cloud, shape))
        self.room = cloud == "room"
        self.noise = 0.0004 if self.room else 0.0 if cloud == "sphere" else 0.001
        self.prims = []

        def add(kind, centre, rot, params):
            self.prims.append((kind, torch.tensor(centre, device="cuda"), torch.tensor(rot, device="cuda"), params))

        def somewhere(d):
            return [r.uniform(-d, d) for _ in range(3)]

        def semi(lo, hi):
            return tuple(r.uniform(lo, hi) for _ in range(3))

        if cloud == "sphere":
            add("ellipsoid", [0.0, 0.0, 0.0], _turn(None), (0.5, 0.5, 0.5))
        elif cloud == "object":
            for _ in range(3):
                add("ellipsoid", somewhere(0.4), _turn(r), semi(0.1, 0.4))
            add("torus", somewhere(0.3), _turn(r), (0.3, 0.08))
        elif cloud == "superquadric":
            for _ in range(10):
                add("superquadric", somewhere(0.5), _turn(r), semi(0.1, 0.4) + (r.uniform(0.3, 3.0), r.uniform(0.3, 3.0)))
        elif cloud == "mixed":
            for _ in range(r.randint(1, 5)):
                kind = r.choice(["ellipsoid", "box", "torus"])
                big = r.uniform(0.15, 0.35)
                add(kind, somewhere(0.4), _turn(r), semi(0.1, 0.4) if kind == "ellipsoid" else
                    semi(0.08, 0.35) if kind == "box" else (big, r.uniform(0.04, 0.4 * big)))
        else:  # room: 10 x 8 x 3 m scaled by 0.2, with 60 boxes and cylinders on the floor
            add("box", [0.0, 0.0, 0.0], _turn(None), (1.0, 0.8, 0.3))
            for _ in range(60):
                x, y, z = semi(0.02, 0.15)
                c, s = math.cos(a := r.uniform(0, 2 * math.pi)), math.sin(a)
                at = [r.uniform(-0.85, 0.85), r.uniform(-0.65, 0.65), z - 0.3]
                box = r.random() < 0.5
                add("box" if box else "cylinder", at, [[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]],
                    (x, y, z) if box else (x, z))

    def area(self):
        """About the surface's area (parts inside other primitives left out roughly)."""
        total = 0.0
        for kind, _, _, p in self.prims:
            if kind in ("ellipsoid", "superquadric"):
                a, b, c = (x ** 1.6 for x in p[:3])
                total += 4 * math.pi * ((a * b + a * c + b * c) / 3) ** (1 / 1.6)
            elif kind == "torus":
                total += 4 * math.pi ** 2 * p[0] * p[1]
            elif kind == "box":
                total += 8 * (p[0] * p[1] + p[1] * p[2] + p[0] * p[2])
            else:
                total += 4 * math.pi * p[0] * p[1] + 2 * math.pi * p[0] ** 2
        return total * (1.0 if len(self.prims) == 1 or self.room else 0.7)

    def distance(self, x):
        """Approximate signed distance (inside negative; in a room, the free space positive)."""
        out = None
        for k, (kind, c, rot, p) in enumerate(self.prims):
            d = _distance(kind, (x - c) @ rot, p)
            d = -d if self.room and k == 0 else d
            out = d if out is None else torch.minimum(out, d)
        return out

    def sample(self, n, g):
        """n points of the surface, about uniform by area, in random order, with the cloud's noise."""
        areas = [self._area_of(p) for p in self.prims]
        got, count = [], 0
        while count < n:
            want = int(1.5 * (n - count)) + 64
            for k, prim in enumerate(self.prims):
                m = int(want * areas[k] / sum(areas)) + 8
                x = _on_surface(prim, m, g)
                keep = torch.ones(m, dtype=torch.bool, device="cuda")
                for j, (kind, c, rot, p) in enumerate(self.prims):
                    if j != k and not (self.room and j == 0):
                        keep &= _distance(kind, (x - c) @ rot, p) > 0
                x = x[keep]
                got.append(x)
                count += x.shape[0]
        x = torch.cat(got)
        x = x[torch.randperm(x.shape[0], generator=g, device="cuda")[:n]]
        if self.noise:
            x = x + self.noise * torch.randn(x.shape, generator=g, device="cuda")
        return x.clamp(-1.0, 1.0).contiguous()

    def _area_of(self, prim):
        one = Shape.__new__(Shape)
        one.prims, one.room = [prim], False
        return one.area()

    def normals(self, x):
        """Unit gradient of the distance at x."""
        e = 1e-3
        d = torch.stack([self.distance(x + e * a) - self.distance(x - e * a) for a in torch.eye(3, device="cuda")], 1)
        return (d / d.norm(dim=1, keepdim=True).clamp_min(1e-12)).contiguous()


def _turn(r):
    w, x, y, z = (1.0, 0.0, 0.0, 0.0) if r is None else (r.gauss(0, 1) for _ in range(4))
    n = math.sqrt(w * w + x * x + y * y + z * z)
    w, x, y, z = w / n, x / n, y / n, z / n
    return [[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
            [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
            [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]]


def _distance(kind, p, par):
    if kind == "ellipsoid":
        a = torch.tensor(par, device=p.device)
        k0, k1 = (p / a).norm(dim=1), (p / (a * a)).norm(dim=1)
        return k0 * (k0 - 1) / k1.clamp_min(1e-12)
    if kind == "torus":
        return torch.hypot(torch.hypot(p[:, 0], p[:, 1]) - par[0], p[:, 2]) - par[1]
    if kind == "superquadric":
        a, b, c, e1, e2 = par
        xy = (p[:, 0] / a).abs() ** (2 / e2) + (p[:, 1] / b).abs() ** (2 / e2)
        val = xy ** (e2 / e1) + (p[:, 2] / c).abs() ** (2 / e1)
        return p.norm(dim=1) * (1 - val.clamp(1e-12, 1e12) ** (-e1 / 2))
    if kind == "box":
        d = p.abs() - torch.tensor(par, device=p.device)
    else:  # cylinder
        d = torch.stack([torch.hypot(p[:, 0], p[:, 1]) - par[0], p[:, 2].abs() - par[1]], 1)
    return d.clamp_min(0).norm(dim=1) + d.amax(1).clamp_max(0)


def _on_surface(prim, n, g):
    kind, c, rot, par = prim

    def rand(*s):
        return torch.rand(*s, generator=g, device="cuda")

    def resample(x, w):  # n of the candidates, in proportion to their area elements
        cum = w.double().cumsum(0)
        return x[torch.searchsorted(cum, rand(n).double() * cum[-1]).clamp_max(x.shape[0] - 1)]

    if kind == "ellipsoid":
        a = torch.tensor(par, device="cuda")
        u = torch.randn(2 * n, 3, generator=g, device="cuda")
        u = u / u.norm(dim=1, keepdim=True)
        x = resample(u * a, (u / a).norm(dim=1))
    elif kind == "torus":
        th, ph = 2 * math.pi * rand(2 * n), 2 * math.pi * rand(2 * n)
        rr = par[0] + par[1] * ph.cos()
        x = resample(torch.stack([rr * th.cos(), rr * th.sin(), par[1] * ph.sin()], 1), rr)
    elif kind == "superquadric":
        a, b, cc, e1, e2 = par

        def at(u, v):
            s = lambda t, e: t.sign() * t.abs() ** e  # noqa: E731
            eta, om = (u - 0.5) * math.pi, (2 * v - 1) * math.pi
            return torch.stack([a * s(eta.cos(), e1) * s(om.cos(), e2), b * s(eta.cos(), e1) * s(om.sin(), e2),
                                cc * s(eta.sin(), e1)], 1)
        e = 1e-4
        u, v = rand(3 * n).clamp(2 * e, 1 - 2 * e), rand(3 * n).clamp(2 * e, 1 - 2 * e)
        w = torch.linalg.cross(at(u + e, v) - at(u - e, v), at(u, v + e) - at(u, v - e)).norm(dim=1)
        x = resample(at(u, v), w)
    elif kind == "box":
        h = torch.tensor(par, device="cuda")
        w = torch.tensor([par[1] * par[2], par[0] * par[2], par[0] * par[1]], device="cuda")
        axis = torch.searchsorted(w.cumsum(0), rand(n) * w.sum()).clamp_max(2)
        x = (2 * rand(n, 3) - 1) * h
        side = (rand(n) < 0.5).float() * 2 - 1
        x.scatter_(1, axis[:, None], (side * h[axis])[:, None])
    else:  # cylinder
        th, z = 2 * math.pi * rand(n), (2 * rand(n) - 1) * par[1]
        cap = rand(n) * (par[0] + 2 * par[1]) < par[0]
        rr = torch.where(cap, par[0] * rand(n).sqrt(), torch.full_like(z, par[0]))
        x = torch.stack([rr * th.cos(), rr * th.sin(), torch.where(cap, z.sign() * par[1], z)], 1)
    return x @ rot.T + c


# ------------------------------------------------------------------- prepare
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _cloud(shape, n, key, g):
    """The cloud of a case: its points follow from the case (they fix the size of the band), their order from g."""
    pts = shape.sample(n, _generator(key))
    return pts[torch.randperm(n, generator=g, device="cuda")].contiguous()


def _band(ctx, shape, pts, case, g, knn, deterministic=False):
    """A band with mid-fit values and moments; also its slots' coordinates and flags."""
    R = case["R"]
    band = gb.gp_build_band(ctx, pts, R, case.get("M1", 2), case.get("M2", 2), knn, deterministic=deterministic)
    ijk, values, flags = gb.gp_band_export(band)
    for part in torch.arange(band.V_stored, device="cuda").split(1 << 24):
        values[part] = shape.distance(ijk[part].float() * (2.0 / R) - 1.0)
    if case.get("kind") == "mesh":  # a factor of either side: the crossings move, the crossed edges stay
        values *= (0.3 * torch.randn(values.shape, generator=g, device="cuda")).exp()
    else:
        values += (0.2 / R) * torch.randn(values.shape, generator=g, device="cuda")
    values[(flags & 4) == 0] = 0
    gb.gp_band_set_values(band, values)
    _, m, v = _views(band)
    train = (flags & 2) != 0
    m.copy_(torch.where(train, 1e-6 * torch.randn(m.shape, generator=g, device="cuda"), 0.0))
    v.copy_(torch.where(train, 1e-12 * (0.5 + torch.rand(v.shape, generator=g, device="cuda")), 0.0))
    return band, ijk, flags


def _views(band):
    """The band's own arrays (values, moments); each view keeps the band alive."""
    views = gb.gp_band_values(band)
    for x in views:
        x.band = band
    return views


def _spacing(shape, points, k=50):
    """About the distance from a point to its k-th nearest other one."""
    return math.sqrt(k * shape.area() / (math.pi * points))


def _queries(shape, pts, n, g):
    """n queries around points of the cloud, and those points' indices."""
    j = torch.randint(pts.shape[0], (n,), generator=g, device="cuda")
    q = pts[j] + _spacing(shape, pts.shape[0]) * torch.randn(n, 3, generator=g, device="cuda")
    return q.contiguous(), j.int()


def _records(band, shape, pts, n, g):
    q, src = _queries(shape, pts, n, g)
    rec = torch.empty((n, 6), device="cuda")
    gb.gp_nn(band, q, None, rec, hint=src)
    return rec


def prepare(case, seed):
    kind, g = case["kind"], _generator(seed)
    ctx = gb.gp_create(0)
    state = {"case": case, "ctx": ctx}
    if kind == "multi":
        r = random.Random(case["shape"])
        bands, Q, B = [], [], []
        for k in range(case["clouds"]):
            shape = Shape("mixed", 1000 * case["shape"] + k)
            pts = _cloud(shape, _log(r, case["j_min"], case["j_max"]), k, g)
            bands.append(_band(ctx, shape, pts, {"R": r.choice([128, 256, 512])}, g, 50)[0])
            Q.append(10 * pts.shape[0])
            B.append(-(-Q[-1] // 8))
        m = gb.gp_multi_create(ctx, bands, Q, B, seed=int(seed) % (1 << 30), deterministic=case["deterministic"])
        gb.gp_multi_set_step(m, STEP0)
        state.update(multi=m, loss=torch.zeros((len(bands), 8), device="cuda"),
                     values=[_views(b) for b in bands])
        return state
    if kind == "dense":
        R, shape = case["R"], Shape("object", case["shape"])
        pts = shape.sample(max(64, case["B"] // 10), g)
        axis = torch.arange(R + 1, device="cuda").float() * (2.0 / R) - 1.0
        z, y, x = torch.meshgrid(axis, axis, axis, indexing="ij")
        d = shape.distance(torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1))
        d += (0.2 / R) * torch.randn(d.shape, generator=g, device="cuda")
        band = gb.gp_build_band(ctx, pts, R, 0, 0, 0)
        state.update(values=d.contiguous(), rec=_records(band, shape, pts, case["B"], g),
                     grad=torch.empty((R + 1) ** 3, device="cuda"), loss=torch.zeros(8, device="cuda"))
        return state
    shape = Shape(case["cloud"], case["shape"])
    pts = _cloud(shape, case["points"], case["shape"], g)
    if kind == "build":
        state.update(pts=pts)
    elif kind == "fit":
        band, _, _ = _band(ctx, shape, pts, case, g, 50, case["deterministic"])
        state.update(band=band, t=STEP0, fit=FitStep(band, Q=max(10 * case["points"], case["B"]), B=case["B"],
                                                     seed=int(seed) % (1 << 30), weights=WEIGHTS, lr=LR,
                                                     deterministic=case["deterministic"]))
    elif kind == "nn":
        # The search asks for the normals that seed it, which come with the sampling widths.
        band = gb.gp_build_band(ctx, pts, case["R"], 2, 2, 50)
        q, src = _queries(shape, pts, case["queries"], g)
        if case["seeded"]:  # as the sampler emits them: grouped by place
            cell = ((pts[src.long()] + 1) * 32).long().clamp(0, 63)
            key = sum(((cell[:, a] >> b) & 1) << (3 * b + a) for a in range(3) for b in range(6))
            order = key.argsort(stable=True)
            q, src = q[order].contiguous(), src[order].contiguous()
        n = case["queries"]
        state.update(band=band, pts=pts, q=q, hint=src if case["seeded"] else None,
                     nn=torch.empty(n, dtype=torch.int32, device="cuda"), rec=torch.empty((n, 6), device="cuda"),
                     nvalid=torch.zeros(1, dtype=torch.int32, device="cuda"))
    elif kind in ("step", "autograd"):
        det = case.get("deterministic", False)
        band, ijk, flags = _band(ctx, shape, pts, case, g, 50, det)
        rec = _records(band, shape, pts, case["B"], g)
        state.update(band=band, ijk=ijk, flags=flags, rec=rec, loss=torch.zeros(8, device="cuda"))
        if kind == "autograd":
            state["values"] = _views(band)[0].clone().requires_grad_(True)
        elif det:
            state["t"] = STEP0 + 1
        else:
            state["grad"] = torch.empty(band.V_stored, device="cuda")
    else:  # mesh
        band, _, _ = _band(ctx, shape, pts, case, g, 0)
        ref = shape.sample(case["reference"], g)
        state.update(band=band, ref=ref, ref_nrm=shape.normals(ref))
    return state


# ----------------------------------------------------------------------- run
def run(s):
    kind = s["case"]["kind"]
    if kind == "fit":
        fit, t, k = s["fit"], s["t"], s["case"]["steps"]
        loss = fit.run(t) if k == 1 else fit.run_pipelined(t, k)
        s["t"] = t + k
        d, m, v = _views(s["band"])
        return {"loss": loss, "values": d, "m": m, "v": v}
    if kind == "multi":
        gb.gp_multi_step(s["multi"], s["loss"], WEIGHTS, lr=LR)
        return {"loss": s["loss"], "state": s["values"]}
    if kind == "nn":
        gb.gp_nn(s["band"], s["q"], s["nn"], s["rec"], hint=s["hint"], nvalid_out=s["nvalid"])
        return {"nn": s["nn"], "rec": s["rec"], "nvalid": s["nvalid"]}
    if kind == "step":
        if s["case"]["deterministic"]:
            gb.gp_step_update(s["band"], s["rec"], s["case"]["B"], s["loss"], LR, s["t"], WEIGHTS,
                              flags=gb.GP_STEP_DETERMINISTIC)
            s["t"] += 1
            d, m, v = _views(s["band"])
            return {"loss": s["loss"], "values": d, "m": m, "v": v}
        gb.gp_step(s["band"], s["rec"], s["case"]["B"], s["grad"], s["loss"], WEIGHTS)
        return {"loss": s["loss"], "grad": s["grad"]}
    if kind == "autograd":
        x = s["values"]
        x.grad = None
        loss = gridpull_loss(x, s["band"], s["rec"], weights=WEIGHTS)
        loss.backward()
        return {"loss": loss, "grad": x.grad}
    if kind == "dense":
        gb.gp_step_dense_noalloc(s["ctx"], s["case"]["R"], s["values"], s["rec"], s["case"]["B"], s["grad"], s["loss"],
                                 WEIGHTS)
        return {"loss": s["loss"], "grad": s["grad"]}
    if kind == "build":
        c = s["case"]
        band = gb.gp_build_band(s["ctx"], s["pts"], c["R"], c["M1"], c["M2"], c["knn"])
        ijk, _, flags = gb.gp_band_export(band)
        return {"ijk": ijk, "flags": flags, "sigma": gb.gp_band_sigma(band)}
    tri, cells = gb.gp_mesh_extract(s["band"], 0.0)
    got = metrics.surface_metrics(s["ctx"], tri, s["ref"], s["ref_nrm"])
    got["fscore"] = list(got["fscore"].values())
    return {"tri": tri, "cells": cells, "metrics": got}


# ---------------------------------------------------------------------- work
def _band_size(area, R, M):
    """About the vertices of a band of M cells around a surface, which crosses
    about 1.5 area / h^2 cells and is as thick as the dilation."""
    if M < 0:
        return (R + 1) ** 3
    return min((R + 1) ** 3, 1.25 * area * (R / 2) ** 2 * (2 * M + 2))


def work(case):
    kind = case["kind"]
    if kind == "multi":
        r = random.Random(case["shape"])
        total = {"bytes": 0.0, "flops": 0.0}
        for k in range(case["clouds"]):
            j = _log(r, case["j_min"], case["j_max"])
            one = {"kind": "fit", "points": j, "R": r.choice([128, 256, 512]), "M1": 2, "M2": 2, "B": -(-10 * j // 8),
                   "steps": 1}
            w = _fit_work(one, Shape("mixed", 1000 * case["shape"] + k).area())
            total = {n: total[n] + w[n] for n in total}
        return total
    if kind == "dense":
        # The record, the values of the cells it touches (at most the grid) and the whole gradient.
        n = (case["R"] + 1) ** 3
        return {"bytes": 24.0 * case["B"] + 4.0 * min(n, 16 * case["B"]) + 4.0 * n, "flops": 400.0 * case["B"]}
    area = Shape(case["cloud"], case["shape"]).area()
    if kind == "fit":
        return _fit_work(case, area)
    if kind == "nn":
        # Query, source index, index and record of each query; the cloud once.
        n = case["queries"]
        return {"bytes": (44.0 if case["seeded"] else 40.0) * n + 12.0 * case["points"], "flops": 100.0 * n}
    V = _band_size(area, case["R"], max(case["M1"], case["M2"]) if min(case["M1"], case["M2"]) >= 0 else -1)
    if kind == "step":
        # Records once; values read and gradient written, or the update's arrays.
        return {"bytes": 24.0 * case["B"] + (24.0 if case["deterministic"] else 8.0) * V,
                "flops": 400.0 * case["B"] + 40.0 * V}
    if kind == "autograd":
        # The loss needs the records and the values, the gradient a write.
        return {"bytes": 24.0 * case["B"] + 8.0 * V, "flops": 400.0 * case["B"] + 40.0 * V}
    if kind == "build":
        # The cloud in, widths out; coordinates and flags of the band's vertices.
        return {"bytes": 16.0 * case["points"] + 13.0 * V, "flops": 8.0 * 50 * case["points"]}
    # Values once, about 2.5 triangles a crossed cell with their cells; the reference points and their normals.
    crossed = 1.5 * area * (case["R"] / 2) ** 2
    return {"bytes": 4.0 * V + 44.0 * 2.5 * crossed + 24.0 * case["reference"],
            "flops": 100.0 * (16 * 2.5 * crossed + case["reference"])}


def _fit_work(case, area):
    """One step: the cloud's points and widths, a record a query, and on each trainable vertex the value, the gradient
    and the moments that Adam reads and writes."""
    V = _band_size(area, case["R"], max(case["M1"], case["M2"]) if min(case["M1"], case["M2"]) >= 0 else -1)
    return {"bytes": case["steps"] * (16.0 * min(case["points"], case["B"]) + 24.0 * case["B"] + 24.0 * V),
            "flops": case["steps"] * (500.0 * case["B"] + 50.0 * V)}


# --------------------------------------------------------------------- exact
def exact(case, seed):
    """64-bit results in plain torch, from the inputs that prepare() makes (records, values, moments and the storage
    order are inputs here).  None where the whole call draws its own queries."""
    kind = case["kind"]
    if kind == "nn":
        if case["queries"] * case["points"] > 3e11:
            return None
        s = prepare(case, seed)
        nn, pts = _brute_nearest(s["q"], s["pts"]), s["pts"].double()
        return {"nn": None, "rec": torch.cat([s["q"].double(), pts[nn]], 1), "nvalid": None}
    if kind == "build":
        if case["points"] > 150_000:
            return None
        pts, k = prepare(case, seed)["pts"].double(), min(case["knn"], case["points"] - 1)
        sigma = torch.cat([_pair_distances(q, pts).topk(k + 1, dim=1, largest=False).values[:, -1]
                           for q in pts.split(2048)])
        return {"ijk": None, "flags": None, "sigma": sigma}
    if kind not in ("step", "autograd", "dense"):
        return None
    s = prepare(case, seed)
    R = case["R"]
    if kind == "dense":
        n = R + 1
        key = torch.arange(n ** 3, device="cuda")
        ijk = torch.stack([key % n, (key // n) % n, key // (n * n)], 1)
        inner = (ijk < R).all(1)
        L, D = _loss(s["values"], ijk, torch.full_like(key, 4) | (8 * inner.long()), R, s["rec"], tv=False)
        return {"loss": L, "grad": D.grad}
    values = s["values"].detach() if kind == "autograd" else _views(s["band"])[0]
    L, D = _loss(values, s["ijk"], s["flags"], R, s["rec"])
    if kind == "autograd":
        return {"loss": L[0], "grad": D.grad}
    if not case["deterministic"]:
        return {"loss": L, "grad": D.grad}
    _, m, v = _views(s["band"])
    b1, b2, eps, lr = (float(np.float32(x)) for x in (0.9, 0.999, 1e-8, LR))
    train, g = (s["flags"] & 2) != 0, D.grad
    mm = torch.where(train, b1 * m.double() + (1 - b1) * g, m.double())
    vv = torch.where(train, b2 * v.double() + (1 - b2) * g * g, v.double())
    step = lr * (mm / (1 - b1 ** s["t"])) / ((vv / (1 - b2 ** s["t"])).sqrt() + eps)
    return {"loss": L, "values": torch.where(train, D.detach() - step, D.detach()), "m": mm, "v": vv}


def _pair_distances(q, pts):
    """Distances as differences, not as a product (no cancellation)."""
    d = torch.zeros(q.shape[0], pts.shape[0], dtype=torch.float64, device="cuda")
    for a in range(3):
        d += (q[:, a, None] - pts[None, :, a]) ** 2
    return d.sqrt()


def _brute_nearest(q, pts):
    q, pts = q.double(), pts.double()
    step = max(1, int(2e8 // pts.shape[0]))
    return torch.cat([_pair_distances(part, pts).argmin(1) for part in q.split(step)])


def _loss(values, ijk, flags, R, rec, tv=True):
    """The loss slots and the values with their gradient, all in 64 bits."""
    D = values.detach().double().requires_grad_(True)
    n1, ijk, flags = R + 1, ijk.long(), flags.long()
    slot = torch.full((n1 ** 3,), -1, dtype=torch.int64, device="cuda")
    there = (flags & 4) != 0
    key = ijk[:, 0] + n1 * (ijk[:, 1] + n1 * ijk[:, 2])
    slot[key[there]] = torch.nonzero(there)[:, 0]
    x = rec.double()
    inside = torch.isfinite(x).all(1)
    t = (x + 1) * (R / 2)
    c = t.floor()
    inside &= ((c[:, :3] >= 0) & (c[:, :3] <= R - 1)).all(1)
    c = torch.nan_to_num(c).clamp(0, R - 1)
    t, c = t - c, c.long()
    low = [slot[c[:, o] + n1 * (c[:, o + 1] + n1 * c[:, o + 2])] for o in (0, 3)]
    ok = inside & (low[0] >= 0) & (low[1] >= 0)
    for a in low:
        ok &= (flags[a.clamp_min(0)] & 8) != 0
    t, c, x = t[ok], c[ok], x[ok]
    bv = int(ok.sum())

    def field(o):
        f, grad, w = 0.0, [0.0, 0.0, 0.0], t[:, o:o + 3]
        for k in range(8):
            b = (k & 1, (k >> 1) & 1, k >> 2)
            d = D[slot[c[:, o] + b[0] + n1 * (c[:, o + 1] + b[1] + n1 * (c[:, o + 2] + b[2]))]]
            e = [w[:, a] if b[a] else 1 - w[:, a] for a in range(3)]
            f = f + d * e[0] * e[1] * e[2]
            for a in range(3):
                grad[a] = grad[a] + (1 if b[a] else -1) * d * e[(a + 1) % 3] * e[(a + 2) % 3]
        grad = torch.stack(grad, 1) * (R / 2)
        return f, grad / grad.norm(dim=1, keepdim=True).clamp_min(1e-12)

    f, n = field(0)
    fs, ns = field(3)
    r = x[:, :3] - x[:, 3:] - f[:, None] * n
    pull, grad, surf = r.norm(dim=1).sum() / max(bv, 1), (1 - (n * ns).sum(1)).sum() / max(bv, 1), fs.abs().sum() / max(bv, 1)
    total, mean_tv, n_tv = pull + WEIGHTS[1] * surf + WEIGHTS[2] * grad, torch.zeros((), device="cuda").double(), 0
    if tv:
        mine = torch.nonzero((flags & 1) != 0)[:, 0]
        n_tv = mine.numel()
        s2 = torch.zeros(n_tv, dtype=torch.float64, device="cuda")
        for a in range(3):
            for d in (-1, 1):
                p = ijk[mine].clone()
                p[:, a] += d
                fine = (p[:, a] >= 0) & (p[:, a] <= R)
                at = slot[(p[:, 0] + n1 * (p[:, 1] + n1 * p[:, 2])).clamp(0, n1 ** 3 - 1)].clamp_min(0)
                s2 = s2 + torch.where(fine, (D[mine] - D[at]) ** 2, 0.0)
        mean_tv = torch.where(s2 > 0, s2.clamp_min(1e-300).sqrt(), 0.0).sum() / max(n_tv, 1)
        total = total + WEIGHTS[0] * mean_tv
    total.backward()
    L = torch.tensor([float(z) for z in (total, pull, grad, surf, mean_tv, bv, n_tv, 0.0)], dtype=torch.float64,
                     device="cuda")
    return L, D
