"""The work that a user of this library has it do, as measurable cases.

A case is a dict of plain values; `prepare` makes the handles and inputs a program holds
before the call, `run` makes the call through the public binding, `work` states the bytes
and operations the call cannot do without, and `exact` restates the small and medium
results in 64-bit torch, from the definition (extruded convex footprints, rays toward the
sun) and without the library.

Cities, grids and sun tables follow the repository's own workloads: boxes on a 4 x 4 grid,
convex footprints on a street grid with lognormal heights and 30 m wall bands, a park
ringed by towers, one-minute sun steps from 9 to 17 h at 40.7 degrees north.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1907_04435_gb300 import autograd
from paper_1907_04435_gb300 import binding as B

LAT = math.radians(40.7)
STEP_CHOICES = (1.0, 2.0, 4.0)


# ------------------------------------------------------------------------------- cases
def listed():
    return [
        # the smallest study: 16 boxes, a 64 x 64 raster at 2 m, two-minute steps; a call
        # of a few hundred microseconds, as an interactive tool makes after every edit
        dict(name="boxes_map", kind="ground", method="accrual_sam", city="boxes", buildings=16, nx=64, ny=64,
             dx=2.0, doy=172, days=1, step=2.0, closed=True),
        # the same study by the plain per-step ray sweep, the reference method users check against
        dict(name="boxes_sweep", kind="ground", method="sweep_trace", city="boxes", buildings=16, nx=64, ny=64,
             dx=2.0, doy=172, days=1, step=2.0, closed=False),
        # the ground of a whole district for one day: the ordinary large call
        dict(name="district_ground", kind="ground", method="accrual_sam", city="district", buildings=2000,
             nx=2048, ny=2048, dx=1.0, doy=172, days=1, step=1.0, closed=True),
        # the facades of the same district: a million wall samples with normals
        dict(name="district_facades", kind="points", method="accrual_sam", city="district", buildings=2000,
             n=1_000_000, doy=172, days=1, step=1.0, closed=True),
        # the ray-traced accrual on part of the district, ragged against every tile size
        dict(name="district_traced", kind="ground", method="accrual_trace", city="district", buildings=2000,
             nx=517, ny=389, dx=1.0, doy=172, days=1, step=1.0, closed=False),
        # one lot and its surroundings over a season, from a mesh nobody declared closed
        dict(name="lot_season", kind="ground", method="accrual_sam", city="district", buildings=2000,
             nx=231, ny=187, dx=1.0, doy=172, days=92, step=1.0, closed=False),
        # a season over a large city through the direction graph (one map per sun-path bin)
        dict(name="season_graph", kind="graph", method="accrual_sam", city="district", buildings=50_000,
             nx=1024, ny=1024, dx=1.0, doy=172, days=92, step=1.0, bin_deg=5.0),
        # development variants x intervals in one launch, with a kept plan and kept outputs
        dict(name="scenarios", kind="batch", city="district", buildings=2000, nx=1024, ny=1024, dx=1.0,
             variants=16, intervals=2, doy=172, days=3, step=1.0),
        # gradient of a park's shadow-minutes with respect to the heights around it: new
        # heights, forward and backward
        dict(name="park_gradient", kind="gradient", city="park", buildings=200, nx=1000, ny=600, dx=0.5,
             doy=79, days=1, step=1.0),
        # the approximate inverse accrual map of a neighbourhood
        dict(name="inverse_map", kind="ground", method="iam", city="district", buildings=2000, nx=613, ny=457,
             dx=1.0, doy=172, days=1, step=1.0, closed=True),
        # which buildings shadow a square: per-building areas over a polygon
        dict(name="contribution", kind="contribution", city="district", buildings=2000, nx=512, ny=512, dx=1.0,
             doy=172, days=1, step=1.0),
        # a serving request: host mesh, sun and wall samples in, host counts out
        dict(name="request", kind="request", city="district", buildings=500, n=100_000, nx=600, ny=500, dx=1.0,
             doy=172, days=1, step=2.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("map", "map", "sweep", "facades", "traced", "season", "graph", "batch", "gradient", "iam",
                       "contribution", "request"))
    c = dict(city="district", dx=rng.choice((0.5, 1.0, 2.0, 2.5)), doy=rng.randint(1, 365), days=1,
             step=rng.choice(STEP_CHOICES))
    if kind == "map":
        c.update(kind="ground", method="accrual_sam", buildings=_log_int(rng, 16, 4000), nx=_log_int(rng, 33, 2000),
                 ny=_log_int(rng, 33, 2000), days=rng.randint(1, 2), closed=rng.random() < 0.7, dx=rng.choice((1.0, 2.0)))
    elif kind == "sweep":
        c.update(kind="ground", method=rng.choice(("sweep_trace", "sweep_raster")), buildings=_log_int(rng, 16, 500),
                 nx=_log_int(rng, 33, 300), ny=_log_int(rng, 33, 300), closed=False, step=rng.choice((2.0, 4.0)))
    elif kind == "facades":
        c.update(kind="points", method=rng.choice(("accrual_sam", "accrual_sam", "accrual_trace")),
                 buildings=_log_int(rng, 50, 4000), closed=rng.random() < 0.7)
        c["n"] = _log_int(rng, 1000, 1_000_000 if c["method"] == "accrual_sam" else 50_000)
    elif kind == "traced":
        c.update(kind="ground", method="accrual_trace", buildings=_log_int(rng, 50, 4000), nx=_log_int(rng, 40, 500),
                 ny=_log_int(rng, 40, 400), closed=False)
    elif kind == "season":
        c.update(kind="ground", method="accrual_sam", buildings=_log_int(rng, 100, 2000), nx=_log_int(rng, 60, 250),
                 ny=_log_int(rng, 60, 250), days=rng.randint(7, 92), closed=rng.random() < 0.5, dx=1.0)
    elif kind == "graph":
        c.update(kind="graph", method="accrual_sam", buildings=_log_int(rng, 500, 50_000), nx=_log_int(rng, 100, 1000),
                 ny=_log_int(rng, 100, 1000), dx=1.0, days=rng.randint(14, 92), doy=172, step=rng.choice((1.0, 2.0)),
                 bin_deg=rng.choice((3.0, 5.0)))
    elif kind == "batch":
        c.update(kind="batch", buildings=_log_int(rng, 300, 2000), nx=_log_int(rng, 300, 1000),
                 ny=_log_int(rng, 300, 1000), dx=1.0, variants=rng.randint(1, 12), intervals=rng.randint(1, 2),
                 doy=rng.choice((79, 172, 266)), days=rng.randint(1, 3), step=rng.choice((1.0, 2.0)))
    elif kind == "gradient":
        c.update(kind="gradient", city="park", buildings=_log_int(rng, 40, 200), nx=_log_int(rng, 60, 1000),
                 ny=_log_int(rng, 60, 600), dx=0.5)
    elif kind == "iam":
        c.update(kind="ground", method="iam", buildings=_log_int(rng, 50, 2000), nx=_log_int(rng, 40, 600),
                 ny=_log_int(rng, 40, 400), closed=True, doy=rng.randint(80, 260))
    elif kind == "contribution":
        c.update(kind="contribution", buildings=_log_int(rng, 50, 2000), nx=_log_int(rng, 40, 500),
                 ny=_log_int(rng, 40, 500), dx=1.0, doy=rng.randint(80, 260))
    else:
        c.update(kind="request", buildings=_log_int(rng, 50, 1000), n=_log_int(rng, 1000, 100_000),
                 nx=_log_int(rng, 60, 800), ny=_log_int(rng, 60, 600))
    return c


# ------------------------------------------------------------------------------ inputs
def _rng(seed, salt):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, salt])


def _convex(rng, n, nv):
    """n sorted rows of nv angles whose gaps make a convex polygon around the centre."""
    out = np.empty((n, nv))
    todo = np.arange(n)
    while todo.size:
        a = np.sort(rng.uniform(0.0, 2 * math.pi, (todo.size, nv)), axis=1)
        gaps = np.diff(np.concatenate([a, a[:, :1] + 2 * math.pi], axis=1), axis=1)
        ok = (gaps.min(axis=1) > 0.25) & (gaps.max(axis=1) < math.pi - 0.1)
        out[todo[ok]] = a[ok]
        todo = todo[~ok]
    return out


class _City:
    """Footprints grouped by vertex count: self.groups is a list of (ids, xy [m, v, 2])."""

    def __init__(self, case, seed):
        rng = _rng(seed, 1)
        n = int(case["buildings"])
        if case["city"] == "boxes":
            side = max(1, int(math.ceil(math.sqrt(n))))
            i, j = np.arange(n) % side, np.arange(n) // side
            s = rng.uniform(20.0, 40.0, (n, 2)) / 2
            c = np.stack([i * 55.0 + 20.0, j * 55.0 + 20.0], 1)
            q = np.array([[-1, -1], [1, -1], [1, 1], [-1, 1]], float)
            self.groups = [(np.arange(n), c[:, None, :] + q[None] * s[:, None, :])]
            self.heights = rng.uniform(10.0, 100.0, n).astype(np.float32)
            self.band, self.extent = 0.0, (side * 55.0 - 15.0, side * 55.0 - 15.0)
            return
        self.band = 30.0
        hole = None
        if case["city"] == "park":
            w, d = case["nx"] * case["dx"], case["ny"] * case["dx"]
            lo, hi, median = (-300.0, -300.0), (w + 300.0, d + 300.0), 60.0
            hole = (w, d)
        else:
            e = max(300.0, 2048.0 * math.sqrt(n / 2000.0))
            lo, hi, median = (0.0, 0.0), (e, e), 30.0
        lots = self._lots(lo, hi)
        if hole is not None:
            x0, y0, x1, y1 = lots.T
            lots = lots[~((x1 > -18) & (x0 < hole[0] + 18) & (y1 > -18) & (y0 < hole[1] + 18))]
        n = min(n, len(lots))
        lots = lots[np.sort(rng.choice(len(lots), n, replace=False))]
        half = rng.uniform(0.6, 1.0, (n, 1)) * ((lots[:, 2:] - lots[:, :2]) / 2 - 1.0)
        centre = (lots[:, 2:] + lots[:, :2]) / 2
        nv = rng.integers(4, 9, n)
        self.groups = []
        for v in range(4, 9):
            ids = np.nonzero(nv == v)[0]
            if ids.size:
                a = _convex(rng, ids.size, v)
                xy = centre[ids, None] + half[ids, None] * np.stack([np.cos(a), np.sin(a)], -1)
                self.groups.append((ids, xy))
        self.heights = np.minimum(rng.lognormal(math.log(median), 0.8, n), 400.0).astype(np.float32)
        self.extent = (hi[0], hi[1])

    @staticmethod
    def _lots(lo, hi):
        """80 x 250 m blocks with 18 m streets, 2 x 8 lots each."""
        out = []
        nbx = max(1, int((hi[0] - lo[0] + 18) // 98))
        nby = max(1, int((hi[1] - lo[1] + 18) // 268))
        bx, by, cx, cy = np.meshgrid(np.arange(nbx), np.arange(nby), np.arange(2), np.arange(8), indexing="ij")
        x = lo[0] + bx * 98.0 + cx * 40.0
        y = lo[1] + by * 268.0 + cy * 31.25
        return np.stack([x, y, x + 40.0, y + 31.25], -1).reshape(-1, 4)

    @property
    def n(self):
        return len(self.heights)

    def footprints(self):
        f = [None] * self.n
        for ids, xy in self.groups:
            for i, p in zip(ids, xy.astype(np.float32)):
                f[i] = p
        return f

    def mesh(self):
        """Closed prisms, counter-clockwise from outside: vertices, triangles, building ids."""
        verts, tris, tb, base = [], [], [], 0
        for ids, xy in self.groups:
            m, v = xy.shape[:2]
            h = self.heights[ids]
            nb = np.maximum(1, np.ceil(h / self.band).astype(int)) if self.band else np.ones(m, int)
            ring_b = np.repeat(np.arange(m), nb + 1)
            first = np.concatenate([[0], np.cumsum(nb + 1)])
            k = np.arange(len(ring_b)) - first[ring_b]
            z = np.where(k == nb[ring_b], h[ring_b], h[ring_b] * (k / nb[ring_b]).astype(np.float32)).astype(np.float32)
            p = np.concatenate([xy.astype(np.float32)[ring_b], np.repeat(z[:, None, None], v, 1)], 2)
            verts.append(p.reshape(-1, 3))
            low = np.nonzero(k < nb[ring_b])[0]
            i = np.arange(v)
            a = base + low[:, None] * v + i
            b = base + low[:, None] * v + (i + 1) % v
            wall = np.stack([np.stack([a, b, b + v], -1), np.stack([a, b + v, a + v], -1)], 2)
            tris.append(wall.reshape(-1, 3))
            tb.append(np.repeat(ids[ring_b[low]], 2 * v))
            q = np.arange(1, v - 1)
            for rings, up in ((first[1:] - 1, True), (first[:-1], False)):
                o = base + rings[:, None] * v
                f = (o + q, o + q + 1) if up else (o + q + 1, o + q)
                tris.append(np.stack([np.broadcast_to(o, f[0].shape), f[0], f[1]], -1).reshape(-1, 3))
                tb.append(np.repeat(ids, v - 2))
            base += len(ring_b) * v
        return np.concatenate(verts), np.concatenate(tris).astype(np.int32), np.concatenate(tb).astype(np.int32)

    def facades(self, n, seed):
        """n wall samples uniform by area: positions and outward normals, float32."""
        rng = _rng(seed, 2)
        a = np.concatenate([xy.reshape(-1, 2) for _, xy in self.groups])
        b = np.concatenate([np.roll(xy, -1, 1).reshape(-1, 2) for _, xy in self.groups])
        h = np.concatenate([np.repeat(self.heights[ids], xy.shape[1]) for ids, xy in self.groups]).astype(float)
        e = b - a
        length = np.hypot(e[:, 0], e[:, 1])
        cum = np.cumsum(length * h)
        k = np.minimum(np.searchsorted(cum, rng.uniform(0, cum[-1], n)), len(h) - 1)
        p = a[k] + rng.uniform(0, 1, (n, 1)) * e[k]
        pos = np.concatenate([p, (rng.uniform(0, 1, n) * h[k])[:, None]], 1).astype(np.float32)
        nrm = np.stack([e[k, 1] / length[k], -e[k, 0] / length[k], np.zeros(n)], 1).astype(np.float32)
        return pos, nrm

    def edges(self, dev):
        """Footprint edges padded to 8 per building (repeats): start and end [n, 8, 2], float64."""
        p = np.zeros((self.n, 8, 2))
        q = np.zeros((self.n, 8, 2))
        for ids, xy in self.groups:
            xy = xy.astype(np.float32).astype(float)
            at = np.minimum(np.arange(8), xy.shape[1] - 1)
            p[ids], q[ids] = xy[:, at], np.roll(xy, -1, 1)[:, at]
        return torch.from_numpy(p).to(dev), torch.from_numpy(q).to(dev)


def _sun(case, doy=None):
    """Directions toward the sun (float32 [S, 3]) and the first step of each day."""
    doy = case["doy"] if doy is None else doy
    n = int(round(8 * 60 / case["step"])) + 1
    hours = 9.0 + np.arange(n) * (case["step"] / 60.0)
    day = (np.arange(case["days"]) + doy - 1) % 365 + 1.0
    g = 2 * math.pi * (day - 1) / 365
    dec = (0.006918 - 0.399912 * np.cos(g) + 0.070257 * np.sin(g) - 0.006758 * np.cos(2 * g)
           + 0.000907 * np.sin(2 * g) - 0.002697 * np.cos(3 * g) + 0.00148 * np.sin(3 * g))[:, None]
    w = np.radians(15.0 * (hours - 12.0))[None]
    d = np.stack([-np.cos(dec) * np.sin(w), np.sin(dec) * math.cos(LAT) - np.cos(dec) * np.cos(w) * math.sin(LAT),
                  np.sin(dec) * math.sin(LAT) + np.cos(dec) * np.cos(w) * math.cos(LAT)], -1)
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    keep = d[..., 2] > math.sin(math.radians(0.5))
    start = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    d = d[keep].astype(np.float32)
    d /= np.linalg.norm(d.astype(np.float64), axis=1, keepdims=True).astype(np.float32)
    return np.ascontiguousarray(d), start


def _grid(case, city):
    if case["city"] == "park":
        x0 = y0 = 0.0
    else:
        x0 = (city.extent[0] - case["nx"] * case["dx"]) / 2
        y0 = (city.extent[1] - case["ny"] * case["dx"]) / 2
    return float(np.float32(x0)), float(np.float32(y0)), float(case["dx"]), int(case["nx"]), int(case["ny"])


def _polygon(case, city):
    """A non-convex study area inside the grid (an L with slanted sides)."""
    x0, y0, dx, nx, ny = _grid(case, city)
    f = np.array([[0.06, 0.08], [0.93, 0.12], [0.88, 0.55], [0.52, 0.5], [0.48, 0.94], [0.1, 0.9]])
    return (np.array([x0, y0]) + f * np.array([nx * dx, ny * dx])).astype(np.float32)


def _weights(case, seed):
    w = _rng(seed, 3).uniform(0.5, 1.5, case["nx"] * case["ny"])
    return torch.from_numpy(w.astype(np.float32)).cuda()


def _sides(case):
    """Side of each variant's square region, in cells."""
    return [min(case["nx"], case["ny"], (256, 333, 512, 768)[v % 4]) for v in range(case["variants"])]


def _variants(case, city, seed):
    """Towers (1 to 5 boxes of 30 to 60 m, 150 to 450 m high) around a site per variant, the
    base buildings they overlap, and a square region of cells around each site."""
    rng = _rng(seed, 4)
    x0, y0, dx, nx, ny = _grid(case, city)
    lo = np.full((city.n, 2), np.inf)
    hi = np.full((city.n, 2), -np.inf)
    for ids, xy in city.groups:
        lo[ids], hi[ids] = xy.min(1), xy.max(1)
    towers, removed, regions = [], [], []
    for side in _sides(case):
        site = rng.uniform(0.2, 0.8, 2) * [nx * dx, ny * dx] + [x0, y0]
        boxes, rem = [], np.zeros(city.n, bool)
        for _ in range(int(rng.integers(1, 6))):
            t = rng.uniform(30.0, 60.0)
            a = site + rng.uniform(-150, 150, 2) - t / 2
            if any((a < q[1] + 2).all() and (a + t > q[0] - 2).all() for q in boxes):
                continue
            boxes.append((a, a + t, rng.uniform(150.0, 450.0)))
            rem |= ((hi >= a - 1) & (lo <= a + t + 1)).all(1)
        soup = []
        for a, b, h in boxes:
            c = np.array([[a[0], a[1]], [b[0], a[1]], [b[0], b[1]], [a[0], b[1]]])
            p = np.concatenate([np.c_[c, np.zeros(4)], np.c_[c, np.full(4, h)]])
            f = [(i, (i + 1) % 4, (i + 1) % 4 + 4) for i in range(4)] + [(i, (i + 1) % 4 + 4, i + 4) for i in range(4)]
            f += [(4, 5, 6), (4, 6, 7), (0, 2, 1), (0, 3, 2)]
            soup.append(p[np.array(f)].reshape(-1, 9))
        towers.append(np.concatenate(soup).astype(np.float32))
        removed.append(np.nonzero(rem)[0].astype(np.int32))
        at = ((site - [x0, y0]) / dx).astype(int) - side // 2
        regions.append((int(np.clip(at[0], 0, nx - side)), int(np.clip(at[1], 0, ny - side)), side, side))
    return towers, removed, np.asarray(regions, np.int32)


# ------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    city = _City(case, seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "request":
        s["mesh"] = city.mesh()
        s["sun_table"] = _sun(case)
        s["points"] = city.facades(case["n"], seed)
        s["grid"] = _grid(case, city)
        s["n"] = city.n
        return s
    if kind == "gradient":
        s["scene"] = B.Scene.from_footprints(city.footprints(), city.heights, city.band)
        # a step of an optimiser: heights moved a little from the built ones
        h = city.heights * _rng(seed, 5).uniform(0.95, 1.05, city.n).astype(np.float32)
        s["heights"] = torch.from_numpy(h).cuda()
        s["weights"] = _weights(case, seed)
    elif kind in ("graph", "batch", "contribution") or case.get("closed"):
        s["scene"] = B.Scene.from_footprints(city.footprints(), city.heights, city.band)
    else:
        v, t, b = city.mesh()
        s["scene"] = B.Scene(v, t, b, city.n)
    if kind == "points":
        s["recv"] = B.Receivers.points(*city.facades(case["n"], seed))
    else:
        s["recv"] = B.Receivers.ground_grid(*_grid(case, city))
    if kind == "batch":
        s["suns"] = [B.Sun(*_sun(case, case["doy"] + 94 * i)) for i in range(case["intervals"])]
        s["batch"] = B.Batch(s["scene"], s["recv"], *_variants(case, city, seed), s["suns"])
        s["out"] = [torch.zeros(max(1, s["batch"].n_out), dtype=torch.int32, device="cuda") for _ in range(2)]
    else:
        s["sun"] = B.Sun(*_sun(case))
    if kind == "contribution":
        s["polygon"] = _polygon(case, city)
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind in ("ground", "points"):
        return B.sa_accumulate(s["scene"], s["recv"], s["sun"], c["step"], c["method"])
    if kind == "graph":
        return B.sa_accumulate_graph(s["scene"], s["recv"], s["sun"], c["step"], c["method"], bin_deg=c["bin_deg"])
    if kind == "batch":
        return s["batch"].run(*s["out"])
    if kind == "gradient":
        h = s["heights"].detach().requires_grad_()
        S = autograd.shadow_minutes(h, s["scene"], s["recv"], s["sun"], c["step"], s["weights"])
        S.backward()
        return S.detach(), h.grad
    if kind == "contribution":
        return B.sa_building_contribution(s["scene"], s["recv"], s["sun"], s["polygon"])
    # request: everything from host arrays, and the counts back on the host
    scene = B.Scene(*s["mesh"], s["n"], closed=True)
    sun = B.Sun(*s["sun_table"])
    walls = B.Receivers.points(*s["points"])
    ground = B.Receivers.ground_grid(*s["grid"])
    out = [B.sa_accumulate(scene, r, sun, c["step"], "accrual_sam") for r in (ground, walls)]
    return [[t.cpu() for t in o] for o in out]


def work(case):
    """Inputs once, outputs once; one coverage test (three edges, two multiply-adds each) for
    every receiver and step."""
    tri = 12 if case["city"] == "boxes" else 31
    S = case["days"] * (int(round(480 / case["step"])) + 1) * case.get("intervals", 1)
    R = 0 if case["kind"] == "points" else case["nx"] * case["ny"]
    n = case.get("n", 0)
    cells = R + n
    if case["kind"] == "batch":
        cells = sum(side * side for side in _sides(case))
    out = cells * (8 * case["intervals"] if case["kind"] == "batch" else 12)
    if case["kind"] in ("gradient", "contribution"):
        out = 16 * case["buildings"]
    read = case["buildings"] * tri * 36 + S * 12 + n * 24 + (4 * R if case["kind"] == "gradient" else 0)
    return {"bytes": float(read + out), "flops": 12.0 * cells * S}


# -------------------------------------------------------------------- 64-bit definition
def _entry(p, q, h, px, py, pz, ux, uy):
    """Height interval [zlo, zhi] over which the ray p + (z - pz) u is inside each prism."""
    cx, cy = q[..., 0] - p[..., 0], q[..., 1] - p[..., 1]
    a = cx * (py - p[..., 1]) - cy * (px - p[..., 0])
    bc = cx * uy - cy * ux
    z = pz - a / torch.where(bc == 0, torch.ones_like(bc), bc)
    inf = float("inf")
    zlo = torch.where(bc > 0, z, torch.where((bc == 0) & (a < 0), inf, -inf)).amax(-1)
    zhi = torch.where(bc < 0, z, inf).amin(-1)
    return torch.maximum(zlo, torch.clamp(pz.squeeze(-1), min=0.0)), torch.minimum(zhi, h)


def _shadow_bits(city, pts, sun, heights, pairs=None):
    """bool [S, R] for receivers pts [R, 3] in spatially compact chunks of 4096 rows; with
    `pairs`, also collects (step, receiver, building) whose status differs at the next step."""
    dev = pts.device
    p, q = city.edges(dev)
    h = torch.from_numpy(heights.astype(np.float64)).to(dev)
    lo, hi = p.amin(1), p.amax(1)
    d = torch.from_numpy(sun.astype(np.float64)).to(dev)
    u = d[:, :2] / d[:, 2:]
    S, R = len(d), len(pts)
    bits = torch.zeros((S, R), dtype=torch.bool, device=dev)
    for r0 in range(0, R, 4096):
        c = pts[r0:r0 + 4096]
        clo, chi = c.amin(0), c.amax(0)
        for s0 in range(0, S, 16):
            us = u[s0:s0 + 17]            # one more, so that neighbouring steps meet in a chunk
            ulo, uhi = us.amin(0), us.amax(0)
            z = torch.clamp(h - clo[2], min=0.0)[:, None]
            near = ((lo - z * torch.clamp(uhi, min=0) <= chi[:2] + 0.01)
                    & (hi - z * torch.clamp(ulo, max=0) >= clo[:2] - 0.01)).all(1).nonzero().squeeze(1)
            for k0 in range(0, len(near), 24):
                b = near[k0:k0 + 24]
                x = c[None, :, None, :, None]
                zlo, zhi = _entry(p[b], q[b], h[b], x[..., 0, :], x[..., 1, :], x[..., 2, :],
                                  us[:, None, None, None, 0], us[:, None, None, None, 1])
                inside = zlo <= zhi
                bits[s0:s0 + 16, r0:r0 + 4096] |= inside[:16].any(2)
                if pairs is not None:
                    j, r, k = (inside[1:] != inside[:-1]).nonzero(as_tuple=True)
                    pairs.append(torch.stack([s0 + j, r0 + r, b[k]], 1))
    return bits


def _counts(bits, day_start, step):
    gross = bits.sum(0, dtype=torch.int32)
    best = torch.zeros_like(gross)
    for a, b in zip(day_start[:-1], day_start[1:]):
        run = torch.zeros_like(gross)
        for j in range(a, b):
            run = (run + 1) * bits[j]
            best = torch.maximum(best, run)
    return gross, gross.double() * step, best


def _centres(case, city):
    """Cell centres in blocks of 64 x 64 cells, and the place of each in output order."""
    x0, y0, dx, nx, ny = _grid(case, city)
    f = np.float32
    x = (f(x0) + (np.arange(nx, dtype=f) + f(0.5)) * f(dx)).astype(np.float64)
    y = (f(y0) + (np.arange(ny, dtype=f) + f(0.5)) * f(dx)).astype(np.float64)
    iy, ix = np.divmod(np.arange(nx * ny), nx)
    order = np.lexsort((ix, iy, ix // 64, iy // 64))
    pts = np.stack([x[ix], y[iy], np.zeros(nx * ny)], 1)[order]
    return torch.from_numpy(pts).cuda(), torch.from_numpy(order).cuda()


def _ordered(values, order):
    return [torch.empty_like(v).scatter_(0, order, v) for v in values]


def _gradient(case, city, seed):
    """S and dS/dh: the sun moves on the great circle between steps, a status that changes
    over a step does so once, at the last (first) crossing of a building's outline."""
    h32 = city.heights * _rng(seed, 5).uniform(0.95, 1.05, city.n).astype(np.float32)
    sun, _ = _sun(case)
    pts, order = _centres(case, city)
    w = _weights(case, seed).double()[order]
    pairs = []
    bits = _shadow_bits(city, pts, sun, h32, pairs)
    dt = float(case["step"])
    steady = (bits[1:] & bits[:-1]).sum(0, dtype=torch.float64)
    S = (steady * w).sum() * dt
    j, r, b = torch.cat(pairs).T
    keep = bits[j, r] != bits[j + 1, r]
    j, r, b = j[keep], r[keep], b[keep]
    d = torch.from_numpy(sun.astype(np.float64)).cuda()
    d = d / d.norm(dim=1, keepdim=True)
    p, q = city.edges(d.device)
    p, q = p[b], q[b]
    h = torch.from_numpy(h32.astype(np.float64)).cuda()
    hb, x, y = h[b], pts[r, 0, None], pts[r, 1, None]
    z0 = torch.zeros_like(x)
    va, vb = d[j], d[j + 1]
    th = torch.atan2(torch.linalg.cross(va, vb).norm(dim=1), (va * vb).sum(1))

    def at(al):
        wa, wb = torch.sin((1 - al) * th) / torch.sin(th), torch.sin(al * th) / torch.sin(th)
        return wa[:, None] * va + wb[:, None] * vb

    def inside(al):
        v = at(al)
        zlo, zhi = _entry(p, q, hb, x, y, z0, v[:, :1] / v[:, 2:], v[:, 1:2] / v[:, 2:])
        return zlo <= zhi

    one = torch.ones_like(th)
    first = bits[j, r]                     # shadow -> lit
    ok = (inside(0 * one) == first) & (inside(one) != first)
    lo, hi = torch.zeros_like(th), one.clone()
    for _ in range(52):
        mid = (lo + hi) / 2
        same = inside(mid) == first
        lo, hi = torch.where(same, mid, lo), torch.where(same, hi, mid)
    al = (lo + hi) / 2
    # the flip of the union: the last building to leave, the first to arrive
    late = torch.where(first, al, 1 - al)  # shadowed part of the step
    late = torch.where(ok, late, -torch.ones_like(late))
    key, inv = torch.unique(r * (len(sun) - 1) + j, return_inverse=True)
    best = torch.full((len(key),), -1.0, dtype=torch.float64, device=d.device).scatter_reduce_(0, inv, late, "amax")
    S = S + (torch.where(best >= 0, best, 0.5) * w[key // (len(sun) - 1)]).sum() * dt
    flips = (bits[1:] != bits[:-1]).sum(0)
    seen = torch.zeros_like(flips).scatter_add_(0, key // (len(sun) - 1), torch.ones_like(key))
    S = S + ((flips - seen).double() * w).sum() * 0.5 * dt
    win = ok & (late == best[inv])
    # roof edges: A_e + h B_e(al) = 0, so dal/dh = -B_e / (h B_e')
    v = at(al)
    dv = (-th * torch.cos((1 - al) * th) / torch.sin(th))[:, None] * va + (th * torch.cos(al * th) / torch.sin(th))[:, None] * vb
    ux, uy = v[:, 0] / v[:, 2], v[:, 1] / v[:, 2]
    dux = (dv[:, 0] * v[:, 2] - v[:, 0] * dv[:, 2]) / v[:, 2] ** 2
    duy = (dv[:, 1] * v[:, 2] - v[:, 1] * dv[:, 2]) / v[:, 2] ** 2
    cx, cy = (q - p)[..., 0], (q - p)[..., 1]
    bc = cx * uy[:, None] - cy * ux[:, None]
    a = cx * (y - p[..., 1]) - cy * (x - p[..., 0])
    z = torch.where(bc > 0, -a / torch.where(bc == 0, 1.0, bc), -1.0)
    zlo, e = z.max(1)
    zhi = torch.where(bc < 0, -a / torch.where(bc == 0, 1.0, bc), float("inf")).amin(1)
    tol = 1e-6 * (hb + 1)
    roof = win & (zlo > 0) & ((zlo - hb).abs() <= tol) & (zhi >= hb - tol)
    bce = bc.gather(1, e[:, None]).squeeze(1)
    dbe = (cx.gather(1, e[:, None]).squeeze(1) * duy - cy.gather(1, e[:, None]).squeeze(1) * dux)
    g = torch.where(roof & (dbe != 0), -bce / (hb * dbe), 0.0) * dt * w[r] * torch.where(first, 1.0, -1.0)
    return S, torch.zeros_like(h).scatter_add_(0, b, g)


def exact(case, seed):
    kind = case["kind"]
    S = case["days"] * (int(round(480 / case["step"])) + 1)
    city = _City(case, seed)
    if kind == "gradient":
        return _gradient(case, city, seed)
    if kind == "ground" and case["method"] != "iam" and case["nx"] * case["ny"] * S <= 1e8:
        sun, start = _sun(case)
        pts, order = _centres(case, city)
        return tuple(_ordered(_counts(_shadow_bits(city, pts, sun, city.heights), start, case["step"]), order))
    if kind == "points" and case["n"] * S <= 2e6:
        sun, start = _sun(case)
        pos, nrm = city.facades(case["n"], seed)
        o = torch.from_numpy(pos.astype(np.float64) + 0.01 * nrm.astype(np.float64)).cuda()
        return _counts(_shadow_bits(city, o, sun, city.heights), start, case["step"])
    return None
