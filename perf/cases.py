"""The work that users have this library do, as cases that can be timed.

A case is one call, or one short chain of calls, of the public entry points
on one part: a block with a pocket (a few thousand triangles), a prismatic
housing (about 200,000 at its usual resolution) or an impeller (up to 1.9
million).  The parts are meshed here, on the GPU; the seed of a case turns
into dimensions a few percent off the nominal ones, a shift, and the sampling
seed, so that two seeds are two different parts of the same triangle list.
"""
from __future__ import annotations

import ctypes
import functools
import math
import random

import numpy as np
import torch

import paper_2609_05467_gb300 as rc

TILT = (12.0, -7.0, 25.0)        # degrees about x, y, z of a part that is not set up along its axes


def listed():
    return [
        # picking a few surface points of a large part in a viewer: the smallest call, and latency is all of it
        dict(name="picked points", path="cast", part="impeller", tris=500_000, points=37, dirs=2048),
        # a small CAD block analysed while it is drawn: every call of the path, launches and waits dominate
        dict(name="pocket block", path="chain", part="pocket", tris=1_472, points=1_000, dirs=256),
        # the housing at its usual sampling: the hemispherical cast that most analyses are made of
        dict(name="housing cast", path="cast", part="housing", tris=203_000, points=100_000, dirs=1024),
        # the largest single part: a finely tessellated impeller, a million points
        dict(name="impeller cast", path="cast", part="impeller", tris=1_930_000, points=1_000_000, dirs=2048),
        # face-level mode: one point at each face centroid, 150 directions (not a multiple of 32), area weights
        dict(name="housing faces", path="faces", part="housing", tris=203_000, points=0, dirs=150),
        # a request of a server or a script: host mesh in, host maps and part result out, in one call
        dict(name="host request", path="host", part="impeller", tris=140_000, points=41_003, dirs=512),
        # loading a large part: acceleration structure and sample points
        dict(name="impeller build", path="build", part="impeller", tris=1_930_000, points=1_000_000, dirs=256),
        # the indicators of a part whose visibility is at hand, with every per-point and per-direction output
        dict(name="indicators", path="indicators", part="housing", tris=203_000, points=300_001, dirs=1000),
        # setup planning of a part in a turned frame: thin rays, covers, and a 6 mm ball-end tool
        dict(name="turned setups", path="setups", part="housing", tris=203_000, points=100_000, dirs=256),
        # finding the machining frame of a part that arrives turned off its axes
        dict(name="turned frame", path="frames", part="housing", tris=203_000, points=100_000, dirs=256),
        # a catalogue of parts of mixed sizes, the whole path of all of them in one launch
        dict(name="catalogue", path="batch", part="mixed", tris=490_000, points=12, dirs=512),
        # a designer moves a bump on one blade: only what the edit can change is cast again
        dict(name="blade edit", path="edit", part="impeller", tris=1_930_000, points=200_000, dirs=1024),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same kinds: sizes over the whole range, most of
    them odd; never more work than the largest listed case."""
    path = rng.choice(["cast", "cast", "cast", "chain", "faces", "host", "build", "indicators", "setups", "frames",
                       "batch", "edit"])
    part = rng.choice(["housing", "impeller"]) if path != "chain" else rng.choice(["pocket", "housing"])
    tris = _log(rng, 2_000, 900_000) if part != "pocket" else rng.choice([46, 184, 1_150, 2_254, 9_200, 36_800])
    dirs = rng.choice([32, 64, 96, 128, 150, 256, 360, 512, 777, 1000, 1024, 2048, 2500, 4096])
    points = _log(rng, 1, 400_000)
    c = dict(path=path, part=part, tris=tris, points=min(points, 800_000_000 // dirs), dirs=dirs)
    if path == "cast":
        c["builder"] = rng.choice([0, 0, 1])            # the clustered tree, for a part that is cast many times
        c["in_order"] = rng.choice([0, 0, 0, 1])        # points already in an order the caller likes
    elif path == "faces":
        c["points"] = 0
        c["dirs"] = min(dirs, 512)
    elif path == "indicators":
        c["conc"] = rng.choice([0, 0, 1])
    elif path in ("setups", "frames"):
        c["points"] = max(points, 500)
    elif path == "batch":
        c.update(part="mixed", tris=_log(rng, 20_000, 400_000), points=rng.randint(2, 16), dirs=min(dirs, 1024))
    elif path == "edit":
        c["part"] = "impeller"
        c["tris"] = max(tris, 20_000)
    return c


# ---------------------------------------------------------------------------
# parts
# ---------------------------------------------------------------------------

def _pocket(k):
    """100 x 60 x 40 mm block with a 30 x 30 x 15 mm pocket in its top; each
    of its 46 rectangles is cut into k x k squares of two triangles."""
    X, Y, Z = (0.0, 35.0, 65.0, 100.0), (0.0, 15.0, 45.0, 60.0), (0.0, 25.0, 40.0)
    rects = []                                                     # corner, edge u, edge v, with u x v outward

    def rect(axis, at, a, b, out):
        """The rectangle a x b of the plane `axis` = at; a, b: intervals of the next two axes in cyclic order."""
        i, j = (axis + 1) % 3, (axis + 2) % 3
        c, u, v = [0.0] * 3, [0.0] * 3, [0.0] * 3
        c[axis], c[i], c[j], u[i], v[j] = at, a[0], b[0], a[1] - a[0], b[1] - b[0]
        rects.append((c, u, v) if out > 0 else (c, v, u))

    xs, ys, zs = ([(q[i], q[i + 1]) for i in range(len(q) - 1)] for q in (X, Y, Z))
    for a in xs:
        for b in ys:
            hole = a == xs[1] and b == ys[1]
            rect(2, Z[1] if hole else Z[2], a, b, 1)
            rect(2, 0.0, a, b, -1)
    for b in zs:
        for a in ys:
            rect(0, X[3], a, b, 1)
            rect(0, 0.0, a, b, -1)
        for a in xs:
            rect(1, Y[3], b, a, 1)
            rect(1, 0.0, b, a, -1)
    for s in (1, -1):
        rect(0, X[1] if s > 0 else X[2], ys[1], zs[1], s)
        rect(1, Y[1] if s > 0 else Y[2], zs[1], xs[1], s)
    V, F = [], []
    for c, u, v in rects:
        c, u, v = (torch.tensor(q, dtype=torch.float64) for q in (c, u, v))
        t = torch.arange(k + 1, dtype=torch.float64) / k
        base = sum(len(q) for q in V)
        V.append((c + t[:, None, None] * u + t[None, :, None] * v).reshape(-1, 3))
        i = (torch.arange(k)[:, None] * (k + 1) + torch.arange(k)[None, :]).reshape(-1) + base
        F += [torch.stack([i, i + k + 1, i + k + 2], 1), torch.stack([i, i + k + 2, i + 1], 1)]
    V, inv = torch.unique(torch.cat(V), dim=0, return_inverse=True)
    return V.cuda(), inv[torch.cat(F)].cuda()


def _housing(x, y, z):
    """Signed function of a 150 x 100 x 50 mm block with a T-slot along x,
    four oblique through-holes and a pocket in each y face."""
    def box(x0, x1, y0, y1, z0, z1):
        return torch.maximum(torch.maximum(torch.maximum(x0 - x, x - x1), torch.maximum(y0 - y, y - y1)),
                             torch.maximum(z0 - z, z - z1))

    far, tilt = 1500.0, math.radians(20.0)
    d = torch.maximum(box(0, 150, 0, 100, 0, 50), -box(-far, far, 44, 56, 40, far))
    d = torch.maximum(d, -box(-far, far, 38, 62, 32, 40))
    for hx in (30.0, 120.0):
        for hy in (20.0, 80.0):
            px, py, pz = x - hx, y - hy, z - 25.0
            s = px * math.sin(tilt) + pz * math.cos(tilt)
            d = torch.maximum(d, 4.0 - torch.sqrt((px - s * math.sin(tilt)) ** 2 + py ** 2
                                                  + (pz - s * math.cos(tilt)) ** 2))
    d = torch.maximum(d, -box(55.5, 94.5, -far, 15, 10, 30))
    return torch.maximum(d, -box(55.5, 94.5, 85, far, 10, 30))


def _impeller(x, y, z):
    """Signed function of a hub of radius 40 mm with twelve twisted blades out to 70 mm, 0.8 mm apart at the tip."""
    beta, gam, pitch = math.radians(90.0) / 30.0, math.radians(35.0) / 30.0, math.pi / 6.0
    thick = 70.0 * pitch / math.sqrt(1.0 + (70.0 * beta) ** 2 + (70.0 * gam) ** 2) - 0.8
    r = torch.sqrt(x * x + y * y)
    hub = torch.maximum(r - 40.0, torch.maximum(-z, z - 40.0))
    turn = ((torch.atan2(y, x) - beta * (z - 5.0) - gam * (r - 40.0)) / pitch + 0.5) % 1.0 - 0.5
    blade = torch.abs(r * turn * pitch / torch.sqrt(1.0 + (r * beta) ** 2 + (r * gam) ** 2)) - thick / 2
    blade = torch.maximum(blade, torch.maximum(r - 70.0, 39.0 - r))
    return torch.minimum(hub, torch.maximum(blade, torch.maximum(5.0 - z, z - 35.0)))


def _march(sdf, lo, hi, h):
    """The zero set of sdf (negative inside) on a grid of spacing h, by marching tetrahedra, wound outward."""
    kw = dict(dtype=torch.float64, device="cuda")
    n = [int(math.ceil((b - a) / h)) + 1 for a, b in zip(lo, hi)]
    ax = [a + h * torch.arange(k, **kw) for a, k in zip(lo, n)]
    f = sdf(ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :])
    corner = [(i, j, k) for i in (0, 1) for j in (0, 1) for k in (0, 1)]
    inside = sum((f[i:n[0] - 1 + i, j:n[1] - 1 + j, k:n[2] - 1 + k] < 0).int() for i, j, k in corner)
    cell = torch.nonzero((inside > 0) & (inside < 8))
    step = torch.tensor([n[1] * n[2], n[2], 1], device="cuda")
    steps = [int(s) for s in (n[1] * n[2], n[2], 1)]
    paths = [[0, steps[a], steps[a] + steps[b], sum(steps)]
             for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1))]      # six tetrahedra along the diagonal
    tet = ((cell * step).sum(1)[:, None, None] + torch.tensor(paths, device="cuda")).reshape(-1, 4)
    out = f.reshape(-1)[tet] >= 0
    tet = torch.gather(tet, 1, torch.argsort(out.int(), dim=1, stable=True))    # inside corners first
    k = 4 - out.sum(1)
    cuts = {1: [((0, 1), (0, 2), (0, 3))], 3: [((0, 3), (1, 3), (2, 3))],
            2: [((0, 2), (0, 3), (1, 3)), ((0, 2), (1, 3), (1, 2))]}
    edge, ends = [], []
    for m in (1, 3, 2):
        t = tet[k == m]
        for cut in cuts[m]:
            edge.append(torch.stack([t[:, list(e)] for e in cut], 1))
            ends.append(t[:, [0, 3]])
    edge, ends = torch.cat(edge).sort(dim=2)[0], torch.cat(ends)
    total = n[0] * n[1] * n[2]
    key, inv = torch.unique(edge[..., 0] * total + edge[..., 1], return_inverse=True)

    def place(g):
        return torch.stack([ax[0][g // steps[0]], ax[1][g // steps[1] % n[1]], ax[2][g % n[2]]], -1)

    a, b = key // total, key % total
    t = (f.reshape(-1)[a] / (f.reshape(-1)[a] - f.reshape(-1)[b]))[:, None]
    V = place(a) + t * (place(b) - place(a))
    e1, e2 = V[inv[:, 1]] - V[inv[:, 0]], V[inv[:, 2]] - V[inv[:, 0]]
    back = (torch.linalg.cross(e1, e2) * (place(ends[:, 1]) - place(ends[:, 0]))).sum(1) < 0
    return V, torch.where(back[:, None], inv.flip(1), inv)


@functools.lru_cache(maxsize=16)
def _nominal(part, tris):
    """(V float64, F int32) of a part at a resolution of about `tris` triangles."""
    if part == "pocket":
        V, F = _pocket(max(1, round(math.sqrt(tris / 92.0))))
    else:
        sdf, lo, hi, h = {"housing": (_housing, (0.0, 0.0, 0.0), (150.0, 100.0, 50.0),
                                      1.67 * math.sqrt(203_000.0 / tris)),
                          "impeller": (_impeller, (-70.0, -70.0, 0.0), (70.0, 70.0, 40.0),
                                       0.69 * math.sqrt(1.93e6 / tris))}[part]
        off = 0.3819660112501051 * h                # no grid point on a face that lies along the axes
        V, F = _march(sdf, [a - 2 * h - off * s for a, s in zip(lo, (1.0, 1.1, 0.9))], [b + 2 * h for b in hi], h)
    return V, F.int().contiguous()


def _turn(deg):
    (ca, sa), (cb, sb), (cc, sc) = ((math.cos(math.radians(d)), math.sin(math.radians(d))) for d in deg)
    return (np.array([[cc, -sc, 0], [sc, cc, 0], [0, 0, 1]]) @ np.array([[cb, 0, sb], [0, 1, 0], [-sb, 0, cb]])
            @ np.array([[1, 0, 0], [0, ca, -sa], [0, sa, ca]]))


def _mesh(part, tris, rng, turn=None):
    V, F = _nominal(part, tris)
    size = torch.tensor([rng.uniform(0.97, 1.03) for _ in range(3)], dtype=torch.float64, device="cuda")
    move = torch.tensor([rng.uniform(-20.0, 20.0) for _ in range(3)], dtype=torch.float64, device="cuda")
    V = V * size
    if turn is not None:
        V = V @ torch.from_numpy(turn.T.copy()).cuda()
    return (V + move).float().contiguous(), F


# ---------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------

class _State:
    """What a user's program holds: arrays, handles (given back when the state goes) and parameters."""

    def __init__(self, **kw):
        self.handles, self.batch = [], None
        self.__dict__.update(kw)

    def build(self, V, F, builder=0):
        h = rc.rc_build_bvh(V, F) if builder == 0 else rc.rc_build_bvh_ex(V, F, builder)
        self.handles.append(h)
        return h

    def sample(self, h, n, weights=False):
        self.P = torch.empty((n, 3), dtype=torch.float32, device="cuda")
        self.N = torch.empty_like(self.P)
        self.face = torch.empty(n, dtype=torch.int32, device="cuda")
        self.weight = torch.empty(n, dtype=torch.float64, device="cuda") if weights else None
        rc.rc_sample_points(h, n, self.p, self.P, self.N, self.face, self.weight)

    def maps(self, n, dirs):
        self.bits = torch.empty((n, (dirs + 31) // 32), dtype=torch.int32, device="cuda")
        self.count = torch.empty(n, dtype=torch.int32, device="cuda")

    def axes(self, n):
        self.mask = torch.empty(n, dtype=torch.uint8, device="cuda")
        self.travel = torch.empty((n, 6), dtype=torch.float32, device="cuda")
        self.cls = torch.empty(n, dtype=torch.uint8, device="cuda")

    def indicators(self, n, dirs):
        self.acc = torch.empty(n, dtype=torch.float32, device="cuda")
        self.conc = torch.empty_like(self.acc)
        self.dom = torch.empty(n, dtype=torch.int8, device="cuda")
        self.dir_area = torch.empty(dirs, dtype=torch.float64, device="cuda")

    def __del__(self):
        if self.batch:
            rc.rc_batch_destroy(self.batch)
        for h in self.handles:
            rc.rc_destroy_bvh(h)


def _plain(x):
    """A result struct as numbers, floating and whole ones apart (padding left out)."""
    real, whole = [], []

    def walk(v):
        if isinstance(v, float):
            real.append(v)
        elif isinstance(v, int):
            whole.append(v)
        elif isinstance(v, ctypes.Array):
            for q in v:
                walk(q)
        elif isinstance(v, ctypes.Structure):
            for f in v._fields_:
                if f[0] not in ("pad", "cast_counters", "ortho_counters"):
                    walk(getattr(v, f[0]))

    walk(x)
    return np.array(real, np.float64), np.array(whole, np.int64)


def prepare(case, seed):
    rng = random.Random(seed)
    path, n, dirs = case["path"], case["points"], case["dirs"]
    frame = _turn(TILT).astype(np.float32).reshape(-1) if path == "setups" else np.eye(3, dtype=np.float32).reshape(-1)
    p = rc.rc_params_default(n_dirs=dirs, seed=rng.getrandbits(32), tool_length=60.0, frame=frame,
                             sample_mode=1 if path == "faces" else 0, always_setups=1,
                             point_order=case.get("in_order", 0), conc_mode=case.get("conc", 0))
    s = _State(path=path, p=p, n=n, dirs=dirs)
    if path == "batch":
        _prepare_batch(s, case, rng)
        return s
    s.V, s.F = _mesh(case["part"], case["tris"], rng, _turn(TILT) if path in ("setups", "frames") else None)
    if path == "faces":
        s.n = n = s.F.shape[0]
    if path == "host":
        s.hV, s.hF = s.V.cpu().pin_memory(), s.F.cpu().pin_memory()
        s.hbits = torch.empty((n, (dirs + 31) // 32), dtype=torch.int32).pin_memory()
        s.hcount = torch.empty(n, dtype=torch.int32).pin_memory()
        s.hmask, s.hcls = (torch.empty(n, dtype=torch.uint8).pin_memory() for _ in range(2))
        return s
    if path in ("build", "chain"):
        s.P = torch.empty((n, 3), dtype=torch.float32, device="cuda")
        s.N = torch.empty_like(s.P)
        s.face = torch.empty(n, dtype=torch.int32, device="cuda")
        s.maps(n, dirs)
        s.axes(n)
        return s
    s.h = s.build(s.V, s.F, case.get("builder", 0))
    s.sample(s.h, n, weights=path in ("faces", "indicators"))
    if path in ("cast", "faces", "indicators", "edit"):
        s.maps(n, dirs)
    if path in ("faces", "indicators"):
        s.indicators(n, dirs)
    if path in ("setups", "frames"):
        s.axes(n)
        s.tool = torch.empty(n, dtype=torch.uint8, device="cuda")
    if path == "indicators":
        rc.rc_hemisphere_cast(s.h, s.P, s.N, p, s.bits, s.count)
        if seed % 2:                          # areas as weights, as in face-level mode, in every other state
            s.weight = torch.rand(n, dtype=torch.float64, device="cuda",
                                  generator=torch.Generator("cuda").manual_seed(seed)) + 0.5
    if path == "edit":
        rc.rc_hemisphere_cast(s.h, s.P, s.N, p, s.bits, s.count)
        lo, hi = s.V.min(0)[0], s.V.max(0)[0]
        mid, a = (lo + hi) / 2, rng.uniform(0.0, 2 * math.pi)
        rad = 0.45 * float((hi - lo)[0])
        at = torch.tensor([float(mid[0]) + rad * math.cos(a), float(mid[1]) + rad * math.sin(a), float(mid[2])],
                          dtype=torch.float64, device="cuda")
        d = (s.V.double() - at).norm(dim=1)
        at = s.V[d.argmin()].double()                                    # a 0.3 mm bump of 4 mm radius on a blade
        d = (s.V.double() - at).norm(dim=1)
        push = torch.where(d < 4.0, (1.0 - (d / 4.0) ** 2) ** 2, 0.0)[:, None] * torch.tensor(
            [-math.sin(a), math.cos(a), 0.0], dtype=torch.float64, device="cuda")
        s.V2 = torch.where(push.abs().sum(1, keepdim=True) > 0, (s.V.double() + 0.3 * push).float(), s.V).contiguous()
        s.changed = torch.empty(s.F.shape[0], dtype=torch.uint8, device="cuda")
        s.P2, s.N2 = torch.empty_like(s.P), torch.empty_like(s.N)
    return s


def _prepare_batch(s, case, rng):
    shape = random.Random(case["tris"])       # which parts: of the case, not of the seed
    s.batch = rc.rc_batch_create(s.p)
    s.parts, plans = [], []
    for k in range(case["points"]):
        part = shape.choice(["pocket", "housing", "impeller"])
        tris = _log(shape, 6_000, case["tris"])
        plans.append((part, tris, min(200_000, _log(shape, 5_000, 120_000))))
    total = sum(q[2] for q in plans)
    s.maps(total, s.dirs)
    at = 0
    for part, tris, n in plans:
        V, F = _mesh(part, tris, rng)
        h = s.build(V, F)
        s.sample(h, n)
        s.parts.append((s.P, s.N, s.face))    # the batch keeps the arrays' addresses
        rc.rc_batch_add_analysis(s.batch, h, s.P, s.N, s.face, s.bits[at:at + n], s.count[at:at + n])
        at += n


def run(s):
    p, path = s.p, s.path
    if path == "cast":
        rc.rc_hemisphere_cast(s.h, s.P, s.N, p, s.bits, s.count)
        return {"bits": s.bits, "count": s.count}
    if path == "faces":
        rc.rc_hemisphere_cast(s.h, s.P, s.N, p, s.bits, s.count)
        m = rc.rc_direction_variability(s.bits, s.N, p, s.weight, s.acc, s.dom, s.conc)
        return {"bits": s.bits, "count": s.count, "acc": s.acc, "dom": s.dom, "conc": s.conc, "part": _plain(m),
                "label": rc.rc_classify(m, p)}
    if path == "chain":
        h = rc.rc_build_bvh(s.V, s.F)
        rc.rc_sample_points(h, s.n, p, s.P, s.N, s.face)
        rc.rc_hemisphere_cast(h, s.P, s.N, p, s.bits, s.count)
        m = rc.rc_direction_variability(s.bits, s.N, p)
        rc.rc_orthogonal_cast(h, s.P, s.N, p, s.mask, s.travel)
        u = rc.rc_min_setups(h, s.mask, s.travel, s.face, p, s.cls)
        rc.rc_destroy_bvh(h)
        return {"P": s.P, "N": s.N, "face": s.face, "bits": s.bits, "count": s.count, "mask": s.mask,
                "travel": s.travel, "cls": s.cls, "part": _plain(m), "label": rc.rc_classify(m, p), "setups": _plain(u)[1]}
    if path == "host":
        r = rc.rc_analyze_part(s.hV, s.hF, s.n, p, s.hbits, s.hcount, s.hmask, s.hcls)
        return {"bits": s.hbits, "count": s.hcount, "mask": s.hmask, "cls": s.hcls, "part": _plain(r)}
    if path == "build":
        h = rc.rc_build_bvh(s.V, s.F)
        rc.rc_sample_points(h, s.n, p, s.P, s.N, s.face)
        rc.rc_destroy_bvh(h)
        return {"P": s.P, "N": s.N, "face": s.face}
    if path == "indicators":
        m = rc.rc_direction_variability(s.bits, s.N, p, s.weight, s.acc, s.dom, s.conc, s.dir_area)
        return {"acc": s.acc, "dom": s.dom, "conc": s.conc, "dir_area": s.dir_area, "part": _plain(m)}
    if path == "setups":
        rc.rc_orthogonal_cast(s.h, s.P, s.N, p, s.mask, s.travel)
        u = rc.rc_min_setups(s.h, s.mask, s.travel, s.face, p, s.cls)
        rc.rc_tool_cast(s.h, s.P, s.N, p, 3.0, 8, s.tool)
        return {"mask": s.mask, "travel": s.travel, "cls": s.cls, "setups": _plain(u)[1], "tool": s.tool}
    if path == "frames":
        f = rc.rc_frame_select(s.h, s.P, s.N, s.face, p, rc.rc_frame_candidates(s.h, p))
        return {"frames": _plain(f)}
    if path == "batch":
        rc.rc_batch_launch(s.batch)
        got = [_plain(r) for r in rc.rc_batch_results(s.batch, len(s.parts))]
        return {"bits": s.bits, "count": s.count, "real": np.stack([g[0] for g in got]),
                "whole": np.stack([g[1] for g in got])}
    rc.rc_refit_bvh(s.h, s.V2)
    moved, box = rc.rc_changed_faces(s.V, s.V2, s.F, s.changed)
    rc.rc_sample_points_on_faces(s.h, p, s.face, s.P2, s.N2)
    rc.rc_hemisphere_update(s.h, s.P2, s.N2, s.face, s.changed, box, p, s.bits, s.count)
    return {"P": s.P2, "N": s.N2, "changed": s.changed, "moved": moved, "bits": s.bits, "count": s.count}


def work(case):
    """Each array that goes in read once, each that comes out written once;
    per hemisphere ray its direction (15 operations) and one triangle test
    (35); per axis ray one triangle test; per visible direction of the
    indicators its direction and sums (25)."""
    path, n, dirs, T = case["path"], case["points"], case["dirs"], case["tris"]
    mesh = 18 * T                                              # 12 bytes a face, 12 bytes a vertex, two faces a vertex
    if path == "faces":
        n = T
    if path == "batch":
        shape, n, mesh = random.Random(T), 0, 0
        for _ in range(case["points"]):
            shape.choice(["pocket", "housing", "impeller"])
            mesh += 18 * _log(shape, 6_000, T)
            n += min(200_000, _log(shape, 5_000, 120_000))
    rows = 4 * n * ((dirs + 31) // 32)
    points, rays = 28 * n, n * dirs
    return {
        "cast": dict(bytes=mesh + 28 * n + rows, flops=50 * rays),
        "faces": dict(bytes=mesh + points + rows + 17 * n, flops=65 * rays),
        "chain": dict(bytes=mesh + 2 * points + rows + 30 * n, flops=65 * rays + 210 * n),
        "host": dict(bytes=mesh + points + rows + 30 * n, flops=65 * rays + 210 * n),
        "batch": dict(bytes=mesh + points + rows + 30 * n, flops=65 * rays + 210 * n),
        "build": dict(bytes=2 * mesh + points, flops=60 * T + 40 * n),
        "indicators": dict(bytes=rows + 29 * n + 8 * dirs, flops=12 * rays),
        "setups": dict(bytes=mesh + points + 30 * n, flops=35 * 15 * n),
        "frames": dict(bytes=mesh + points, flops=35 * 15 * n + 20 * 384 * T / 2),
        "edit": dict(bytes=3 * mesh + 3 * points + T, flops=60 * T + 40 * n),
    }[path]


# ---------------------------------------------------------------------------
# the same numbers in 64 bits
# ---------------------------------------------------------------------------

def _exact_points(s):
    """Points and normals of area sampling: the quantised area prefix and the counter-based draws in numpy."""
    V, F = s.V.cpu().numpy().astype(np.float64), s.F.cpu().numpy().astype(np.int64)
    A, B, C = V[F[:, 0]], V[F[:, 1]], V[F[:, 2]]
    cr = np.cross(B - A, C - A)
    area = 0.5 * np.sqrt((cr * cr).sum(1))
    prefix = np.cumsum(np.rint(area / area.max() * 2.0 ** 32).astype(np.int64))
    golden = np.uint64(0x9E3779B97F4A7C15)

    def u(k):
        with np.errstate(over="ignore"):
            z = (np.uint64(s.p.seed) ^ ((3 * np.arange(s.n, dtype=np.uint64) + np.uint64(k)) * golden)) + golden
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        return ((z ^ (z >> np.uint64(31))) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53

    f = np.searchsorted(prefix, np.floor(u(0) * float(prefix[-1])).astype(np.int64), side="right")
    r, v = np.sqrt(u(1))[:, None], u(2)[:, None]
    return {"P": (1 - r) * A[f] + r * (1 - v) * B[f] + r * v * C[f], "N": cr[f] / (2 * area[f])[:, None], "face": None}


def _exact_indicators(s, weighted, conc_mode):
    """Indicators of visibility bits, directions rebuilt in 64 bits."""
    n, N = s.n, s.dirs
    j = torch.arange(N, dtype=torch.float64, device="cuda")
    z = 1.0 - (j + 0.5) / N
    r, phi = torch.sqrt(1.0 - z * z), j * (math.pi * (3.0 - math.sqrt(5.0)))
    local = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)
    acc, conc = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    area, part = torch.zeros(N, dtype=torch.float64, device="cuda"), torch.zeros(6, dtype=torch.float64, device="cuda")
    for a in range(0, n, 4096):
        b = slice(a, min(n, a + 4096))
        vis = ((s.bits[b, :, None] >> torch.arange(32, device="cuda")) & 1).reshape(-1, s.bits.shape[1] * 32)[:, :N].double()
        q = s.N[b].double()
        x, y, w = q.T
        sg = torch.where(torch.signbit(w), -1.0, 1.0).double()
        k = -1.0 / (sg + w)
        t1 = torch.stack([1.0 + sg * x * x * k, sg * x * y * k, -sg * x], 1)
        t2 = torch.stack([x * y * k, sg + y * y * k, -y], 1)
        d = torch.einsum("jc,pck->pjk", local, torch.stack([t1, t2, q], 1))
        cnt = vis.sum(1)
        M = (d * vis[..., None]).sum(1).abs()
        dom = M.argmax(1)
        lead = (d.abs().argmax(2) == dom[:, None]) * vis
        share = M.gather(1, dom[:, None])[:, 0] if conc_mode else lead.sum(1)
        acc[b], conc[b] = cnt / N, torch.where(cnt > 0, share / cnt.clamp(min=1), 0.0)
        wt = s.weight[b] if weighted else torch.ones_like(cnt)
        area += (vis * wt[:, None]).sum(0)
        seen = cnt > 0
        part += torch.stack([(wt * cnt).sum(), wt.sum(), conc[b].sum(), seen.sum().double(), cnt.sum(),
                             torch.zeros((), dtype=torch.float64, device="cuda")])
    return {"acc": acc, "dom": None, "conc": conc, "dir_area": area, "part": None}


def exact(case, seed):
    if case["path"] not in ("build", "indicators", "setups"):
        return None
    s = prepare(case, seed)
    if case["path"] == "build":
        return _exact_points(s)
    if case["path"] == "indicators":
        return _exact_indicators(s, s.weight is not None, case.get("conc", 0)) if s.n * s.dirs < 4e8 else None
    R = torch.from_numpy(np.array(list(s.p.frame), np.float64).reshape(3, 3)).cuda()   # columns are the frame's axes
    q, box = s.P.double() @ R, s.V.double() @ R
    hi, lo = box.max(0)[0] - q, q - box.min(0)[0]
    return {"mask": None, "travel": torch.stack([hi, lo], 2).reshape(-1, 6), "cls": None, "setups": None, "tool": None}
