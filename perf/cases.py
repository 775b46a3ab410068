"""The workloads that the navigator's speed is measured on.

Every case is one call (or, for the differentiable step, one forward and one
backward) through the package's public entry points, on inputs drawn on the
GPU from a seed: points uniform in the exclusive part of the mother volume (the
toy-detector protocol of Sec. 3.2) and isotropic directions.  `exact` restates
each answer in plain FP64 torch: every solid is given by the crossings of the
line with the (unbounded) planes and quadrics of its surfaces, sorted, and by
a membership test at the middle of each interval between two of them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1312_0816_gb300 as geo
from paper_1312_0816_gb300 import autograd, scenes

F64 = torch.float64
DEV = "cuda"
INF = math.inf
TWO_PI = 2.0 * math.pi

WHAT = {"dist_out": geo.GEO_Q_DIST_OUT, "dist_in": geo.GEO_Q_DIST_IN, "safety_out": geo.GEO_Q_SAFETY_OUT,
        "safety_in": geo.GEO_Q_SAFETY_IN, "contains": geo.GEO_Q_CONTAINS}

# one solid per kind for the per-shape queries (sizes as in the toy scenes)
SOLIDS = {"box": (scenes.BOX, (30.0, 20.0, 40.0)), "tube": (scenes.TUBE, (10.0, 40.0, 50.0)),
          "cone": (scenes.CONE, (40.0, 10.0, 30.0, 20.0, 45.0)),
          "tubs": (scenes.TUBS, (10.0, 40.0, 50.0, 0.3, 4.0)),
          "pcon": (scenes.PCON, scenes.Pcon((-30.0, -25.0, -20.0, 20.0, 25.0, 30.0), (0.0,) * 6,
                                            (25.0, 25.0, 10.0, 10.0, 25.0, 25.0)))}
SOLID_ROT = scenes.euler_zxz(0.4, 0.9, 1.7)
SOLID_TRANS = (5.0, -7.0, 3.0)


def listed():
    return [
        # the smallest basket of the paper's basket-size axis (Fig. 3): latency and launches
        {"name": "basket_16", "op": "step", "scene": "toy40", "grid": False, "mode": 1, "bpoint": False, "n": 16},
        # the paper's own basket: 1024 particles in a box with four boxes (Sec. 3.1)
        {"name": "basket_1024", "op": "step", "scene": "box4", "grid": False, "mode": 1, "bpoint": False, "n": 1024},
        # the toy detector with a large basket: the bench's headline
        {"name": "step_toy", "op": "step", "scene": "toy40", "grid": False, "mode": 1, "bpoint": False, "n": 1 << 20},
        # the same detector all in FP64, a ragged basket, with the boundary points (a validation run)
        {"name": "step_fp64", "op": "step", "scene": "toy40", "grid": False, "mode": 0, "bpoint": True, "n": 100003},
        # a volume of many daughters with the uniform grid
        {"name": "step_grid", "op": "step", "scene": "grid512", "grid": True, "mode": 1, "bpoint": False, "n": 1 << 22},
        # non-convex solids: polycones (out-of-line FP64 code), a ragged basket
        {"name": "step_pcon", "op": "step", "scene": "pcon4", "grid": False, "mode": 1, "bpoint": False, "n": 300007},
        # transport as a scheduler runs it: baskets of 16 to 65536 tracks in 64 logical volumes, one launch
        {"name": "batched", "op": "batched", "volumes": 64, "n": 1 << 22},
        # the differentiable step: forward and backward with geometry gradients
        {"name": "adjoint", "op": "adjoint", "scene": "diff3", "n": 1 << 18},
        # point location and safety in the toy detector
        {"name": "contains", "op": "contains", "scene": "toy40", "mode": 1, "n": 1 << 22},
        {"name": "safety", "op": "safety", "scene": "toy40", "mode": 1, "n": (1 << 21) + 77},
        # step and relocation in a geometry tree, tracks that have crossed boundaries before
        {"name": "world", "op": "world", "world": "toy", "mode": 1, "n": 1 << 20},
        # one solid's DistFromOutside on its own (Fig. 2)
        {"name": "shape_cone", "op": "shape", "solid": "cone", "what": "dist_out", "n": 1 << 20},
    ]


def _log_size(rng, lo, hi):
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n | 1 if rng.random() < 0.7 else n))


def draw(rng):
    """One more case of the same ranges: any of the operations, its scenes and
    options, sizes over their whole range."""
    op = rng.choice(["step", "step", "step", "step", "batched", "adjoint", "contains", "safety", "world", "shape"])
    if op == "step":
        scene = rng.choice(["box4", "toy8", "toy40", "toy40", "diff3", "seg4", "pcon4", "pconm", "grid512", "grid512"])
        grid = scene == "grid512" and rng.random() < 0.7
        mode = 0 if rng.random() < 0.25 else 1
        top = (1 << 16) if mode == 0 or scene == "pconm" else (1 << 18) if scene == "grid512" and not grid else 1 << 20
        return {"op": op, "scene": scene, "grid": grid, "mode": mode, "bpoint": rng.random() < 0.3,
                "n": _log_size(rng, 16, top)}
    if op == "batched":
        return {"op": op, "volumes": rng.randint(2, 64), "n": _log_size(rng, 1 << 12, 1 << 22)}
    if op == "adjoint":
        return {"op": op, "scene": rng.choice(["box4", "toy8", "diff3", "toy40"]), "n": _log_size(rng, 1 << 10, 1 << 18)}
    if op == "contains":
        return {"op": op, "scene": rng.choice(["box4", "toy8", "toy40", "pcon4"]), "mode": rng.choice([1, 1, 1, 0]),
                "n": _log_size(rng, 1 << 10, 1 << 20)}
    if op == "safety":
        return {"op": op, "scene": rng.choice(["box4", "toy8", "toy40", "diff3"]), "mode": rng.choice([1, 1, 2]),
                "n": _log_size(rng, 1 << 10, 1 << 21)}
    if op == "world":
        return {"op": op, "world": rng.choice(["toy", "toy", "pcon"]), "mode": 1, "n": _log_size(rng, 1 << 10, 1 << 19)}
    return {"op": op, "solid": rng.choice(sorted(SOLIDS)), "what": rng.choice(sorted(WHAT)),
            "n": _log_size(rng, 1 << 10, 1 << 20)}


# --------------------------------------------------------------------------
# plain FP64 geometry (inputs and exact answers)
# --------------------------------------------------------------------------
# A solid's parameters are tensors that broadcast against the points (one
# entry per point, or one for all), so that one call takes many daughters.

def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _plane_cross(c, x, u):
    s = (c - x) / torch.where(u == 0, 1.0, u)
    return torch.where(u == 0, INF, s)


def _quadric_cross(a, b, x, u):
    """Both crossings of rho = |a + b z|."""
    r0 = a + b * x[2]
    rs = b * u[2]
    A = u[0] * u[0] + u[1] * u[1] - rs * rs
    B = x[0] * u[0] + x[1] * u[1] - r0 * rs
    C = x[0] * x[0] + x[1] * x[1] - r0 * r0
    D = B * B - A * C
    q = -(B + torch.copysign(torch.sqrt(torch.where(D > 0, D, 1.0)), B))
    s1 = torch.where((D > 0) & (A != 0), q / torch.where(A == 0, 1.0, A), INF)
    s2 = torch.where(D > 0, C / q, INF)
    return [s1, s2]


def _wedge(sphi, dphi):
    return (-torch.sin(sphi), torch.cos(sphi)), (torch.sin(sphi + dphi), -torch.cos(sphi + dphi))


def _wedge_cross(sphi, dphi, x, u):
    out = []
    for nx, ny in _wedge(sphi, dphi):
        out.append(_plane_cross(torch.zeros_like(x[0]), nx * x[0] + ny * x[1], nx * u[0] + ny * u[1]))
    return out


def _wedge_has(sphi, dphi, x):
    (ax, ay), (bx, by) = _wedge(sphi, dphi)
    a, b = ax * x[0] + ay * x[1] >= 0, bx * x[0] + by * x[1] >= 0
    return (dphi >= TWO_PI) | torch.where(dphi <= math.pi, a & b, a | b)


def _lines(kind, p):
    """Outer and inner radius lines (a, b) of a tube or cone."""
    if kind == scenes.CONE:
        return ((0.5 * (p[2] + p[4]), (p[4] - p[2]) / (2 * p[0])), (0.5 * (p[1] + p[3]), (p[3] - p[1]) / (2 * p[0])))
    return (p[1], torch.zeros_like(p[1])), (p[0], torch.zeros_like(p[0]))


def _crossings(kind, p, planes, x, u):
    if kind == scenes.BOX:
        return [_plane_cross(sg * p[k], x[k], u[k]) for k in range(3) for sg in (-1.0, 1.0)]
    if kind == scenes.PCON:
        z, rn, rx = planes
        out = [_plane_cross(zk, x[2], u[2]) for zk in z]
        for k in range(len(z) - 1):
            for r in (rx, rn):
                if r[k] + r[k + 1] > 0:
                    b = (r[k + 1] - r[k]) / (z[k + 1] - z[k])
                    out += _quadric_cross(r[k] - b * z[k], b, x, u)
        return out + _wedge_cross(p[0], p[1], x, u)
    dz = p[0] if kind == scenes.CONE else p[2]
    out = [_plane_cross(-dz, x[2], u[2]), _plane_cross(dz, x[2], u[2])]
    for a, b in _lines(kind, p):
        out += _quadric_cross(a, b, x, u)
    return out + (_wedge_cross(p[3], p[4], x, u) if kind == scenes.TUBS else [])


def _inside(kind, p, planes, x):
    if kind == scenes.BOX:
        return (x[0].abs() <= p[0]) & (x[1].abs() <= p[1]) & (x[2].abs() <= p[2])
    rho = torch.sqrt(x[0] * x[0] + x[1] * x[1])
    if kind == scenes.PCON:
        z, rn, rx = planes
        out = torch.zeros_like(rho, dtype=torch.bool)
        for k in range(len(z) - 1):
            f = (x[2] - z[k]) / (z[k + 1] - z[k])
            out |= (f >= 0) & (f <= 1) & (rho <= rx[k] + (rx[k + 1] - rx[k]) * f) & \
                   (rho >= rn[k] + (rn[k + 1] - rn[k]) * f)
        return out & _wedge_has(p[0], p[1], x)
    dz = p[0] if kind == scenes.CONE else p[2]
    (ao, bo), (ai, bi) = _lines(kind, p)
    out = (x[2].abs() <= dz) & (rho <= ao + bo * x[2]) & (rho >= ai + bi * x[2])
    return out & _wedge_has(p[3], p[4], x) if kind == scenes.TUBS else out


def _along(kind, p, planes, x, u, want, after=0.0):
    """Start of the first interval of the line (s >= 0) whose middle is inside
    (want) or outside the solid; crossings up to `after` are passed over."""
    c = torch.stack(torch.broadcast_tensors(*_crossings(kind, p, planes, x, u)))
    c = torch.where((c > after) & torch.isfinite(c), c, INF).sort(dim=0).values
    lo = torch.zeros_like(c[0])
    out = torch.full_like(lo, INF)
    for k in range(c.shape[0] + 1):
        hi = c[k] if k < c.shape[0] else torch.full_like(lo, INF)
        last = ~torch.isfinite(hi)
        mid = torch.where(last, lo + 1.0, 0.5 * (lo + hi))
        ok = (_inside(kind, p, planes, [x[i] + mid * u[i] for i in range(3)]) & ~last) == want
        out = torch.where(torch.isinf(out) & ok & (hi > lo), lo, out)
        lo = hi
    return out


def _seg(r, z, ar, az, br, bz):
    er, ez = br - ar, bz - az
    l2 = er * er + ez * ez
    f = (((r - ar) * er + (z - az) * ez) / torch.where(l2 > 0, l2, 1.0)).clamp(0.0, 1.0)
    return torch.hypot(ar + f * er - r, az + f * ez - z)


def _safety(kind, p, planes, x, inside):
    """Distance to the boundary from inside (or outside); 0 on the other side.
    Box, tube and cone; None for the others."""
    if kind in (scenes.TUBS, scenes.PCON):
        return None
    here = _inside(kind, p, planes, x)
    if kind == scenes.BOX:
        e = [x[k].abs() - p[k] for k in range(3)]
        far = torch.sqrt(sum(v.clamp(min=0.0) ** 2 for v in e))
        near = -torch.maximum(e[0], torch.maximum(e[1], e[2]))
    else:
        rho, z = torch.sqrt(x[0] * x[0] + x[1] * x[1]), x[2]
        dz = p[0] if kind == scenes.CONE else p[2]
        i1, o1, i2, o2 = (p[1], p[2], p[3], p[4]) if kind == scenes.CONE else (p[0], p[1], p[0], p[1])
        wall = (i1 + i2) > 0
        inner = _seg(rho, z, i1, -dz, i2, dz)
        caps = torch.minimum(_seg(rho, z, i1, -dz, o1, -dz), _seg(rho, z, i2, dz, o2, dz))
        edge = torch.minimum(caps, _seg(rho, z, o1, -dz, o2, dz))
        far = torch.minimum(edge, inner)
        near = torch.minimum(edge, torch.where(wall, inner, INF))
    return torch.where(here, near, 0.0) if inside else torch.where(here, 0.0, far)


class _Volume:
    """A scene's solids as tensors."""

    def __init__(self, scene):
        self.scene = scene
        self.nd = scene.n_daughters
        self.kinds = [int(k) for k in scene.kinds]
        self.rot = _t(scene.rot).reshape(-1, 3, 3)
        self.trans = _t(scene.trans).reshape(-1, 3)
        self.prm = _t(scene.params).reshape(-1, 5)
        self.rad = _t(scene.bounding_radius()) * (1 + 1e-9) + 1e-6 if self.nd else _t(np.zeros(0))
        self.mkind, self.mprm = int(scene.mother_kind), list(_t(scene.mother_params))
        self.mplanes = _t(scene.planes_of(scene.mother_params)) if self.mkind == scenes.PCON else None
        # groups of daughters that one call can take: by kind, polycones one by one
        self.groups = [(k, [j for j in range(self.nd) if self.kinds[j] == k], None) for k in set(self.kinds)
                       if k != scenes.PCON]
        self.groups += [(scenes.PCON, [j], _t(scene.planes_of(scene.params[j]))) for j in range(self.nd)
                        if self.kinds[j] == scenes.PCON]

    def chunks(self, n):
        step = max(1, (1 << 25) // max(1, self.nd))
        return [(a, min(n, a + step)) for a in range(0, n, step)]

    def pairs(self, js, P, D=None):
        """(daughter, point) pairs whose bounding sphere the point (or the
        forward line) meets, with the local coordinates."""
        js = torch.tensor(js, device=DEV)
        w = [P[k][None, :] - self.trans[js, k][:, None] for k in range(3)]
        r2 = (self.rad[js] ** 2)[:, None]
        ww = w[0] * w[0] + w[1] * w[1] + w[2] * w[2]
        if D is None:
            hit = ww <= r2
        else:
            dd = (D[0] * D[0] + D[1] * D[1] + D[2] * D[2])[None, :]
            wd = w[0] * D[0] + w[1] * D[1] + w[2] * D[2]
            hit = (ww <= r2) | ((wd < 0) & (ww * dd - wd * wd <= r2 * dd * (1 + 1e-9)))
        a, i = hit.nonzero(as_tuple=True)
        j = js[a]
        W = torch.stack([P[k][i] - self.trans[j, k] for k in range(3)])
        R = self.rot[j]
        x = [(R[:, 0, k] * W[0] + R[:, 1, k] * W[1] + R[:, 2, k] * W[2]) for k in range(3)]
        u = None if D is None else [(R[:, 0, k] * D[0][i] + R[:, 1, k] * D[1][i] + R[:, 2, k] * D[2][i])
                                    for k in range(3)]
        return j, i, x, u, [self.prm[j, k] for k in range(5)]

    def contains(self, P):
        """-2 outside the mother, -1 exclusive part, else the lowest daughter."""
        n = P[0].numel()
        where = torch.full((n,), -1, dtype=torch.int64, device=DEV)
        for a, b in self.chunks(n):
            Q = [c[a:b] for c in P]
            low = torch.full((b - a,), self.nd, dtype=torch.int64, device=DEV)
            for kind, js, planes in self.groups:
                j, i, x, _, p = self.pairs(js, Q)
                ok = _inside(kind, p, planes, x)
                low.scatter_reduce_(0, i[ok], j[ok], "amin")
            where[a:b] = torch.where(low < self.nd, low, -1)
        return torch.where(_inside(self.mkind, self.mprm, self.mplanes, P), where, -2).to(torch.int32)

    def step(self, P, D, skip=None, entered=None):
        """(step, hit) of tracks inside the mother; skip: the daughter just
        left (-1 none), entered: tracks that start on the mother's surface."""
        n = P[0].numel()
        zero = torch.zeros(n, dtype=F64, device=DEV)
        after = zero if entered is None else torch.where(entered, 1e-7, zero)
        best = _along(self.mkind, self.mprm, self.mplanes, P, D, False, after)
        hit = torch.full((n,), -1, dtype=torch.int64, device=DEV)
        for a, b in self.chunks(n):
            Q, E = [c[a:b] for c in P], [c[a:b] for c in D]
            low = torch.full((b - a,), INF, dtype=F64, device=DEV)
            found = []
            for kind, js, planes in self.groups:
                j, i, x, u, p = self.pairs(js, Q, E)
                late = torch.zeros_like(x[0]) if skip is None else torch.where(skip[a:b][i] == j, 1e-7, 0.0)
                s = _along(kind, p, planes, x, u, True, late)
                low.scatter_reduce_(0, i, s, "amin")
                found.append((i, j, s))
            first = torch.full((b - a,), self.nd, dtype=torch.int64, device=DEV)
            for i, j, s in found:
                ok = s == low[i]
                first.scatter_reduce_(0, i[ok], j[ok], "amin")
            win = low < best[a:b]
            hit[a:b] = torch.where(win, first, hit[a:b])
            best[a:b] = torch.where(win, low, best[a:b])
        return best, hit.to(torch.int32)

    def safety(self, P):
        s = _safety(self.mkind, self.mprm, self.mplanes, P, True)
        for j in range(self.nd):
            w = [P[k] - self.trans[j, k] for k in range(3)]
            x = [sum(self.rot[j, r, k] * w[r] for r in range(3)) for k in range(3)]
            s = torch.minimum(s, _safety(self.kinds[j], list(self.prm[j]), None, x, False))
        return s


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _rand(g, n, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(n, dtype=F64, device=DEV, generator=g)


def _directions(g, n):
    cz, ph = _rand(g, n, -1.0, 1.0), _rand(g, n, 0.0, TWO_PI)
    st = torch.sqrt((1.0 - cz * cz).clamp(min=0.0))
    return [st * torch.cos(ph), st * torch.sin(ph), cz]


def _in_mother(v, g, n):
    mp = [float(c) for c in v.mprm]
    if v.mkind == scenes.BOX:
        return [_rand(g, n, -mp[k], mp[k]) for k in range(3)]
    if v.mkind == scenes.TUBE:
        lo, hi, dz = mp[0], mp[1], mp[2]
    else:   # a polycone: its bounding tube, points outside it are drawn again
        lo, hi, dz = 0.0, float(v.mplanes[2].max()), float(v.mplanes[0].abs().max())
    r, ph = torch.sqrt(_rand(g, n, lo * lo, hi * hi)), _rand(g, n, 0.0, TWO_PI)
    return [r * torch.cos(ph), r * torch.sin(ph), _rand(g, n, -dz, dz)]


def _points(v, g, n, exclusive=True):
    """n points uniform in the mother, or in its exclusive part."""
    parts, have = [], 0
    while have < n:
        P = _in_mother(v, g, int(1.3 * (n - have)) + 256)
        if exclusive:
            keep = v.contains(P) == -1
            P = [c[keep] for c in P]
        parts.append(P)
        have += P[0].numel()
    return [torch.cat([q[k] for q in parts])[:n].contiguous() for k in range(3)]


def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _scene(case):
    return scenes.SCENES[case["scene"]]()


def _world(case):
    return scenes.world_toy() if case["world"] == "toy" else scenes.world_pcon()


def _build_world(tree):
    vols = [geo.geo_build_volume(s) for s in tree.volumes]
    return geo.geo_build_world(vols, tree.child, tree.root)


def _baskets(case):
    return scenes.batched64(seed=3, n_volumes=case["volumes"], total=case["n"])


def _solid(case):
    """The query's solid as the one daughter of a volume."""
    kind, spec = SOLIDS[case["solid"]]
    return _Volume(scenes._scene("one", scenes.BOX, (1.0, 1.0, 1.0), [(kind, spec, SOLID_ROT, SOLID_TRANS)]))


def _inputs(case, seed):
    """Plain tensors of the case, from the seed alone."""
    g = _generator(seed)
    n, op = case["n"], case["op"]
    if op in ("step", "adjoint"):
        v = _Volume(_scene(case))
        return _points(v, g, n) + _directions(g, n) + ([_rand(g, n, -1.0, 1.0)] if op == "adjoint" else [])
    if op in ("contains", "safety"):
        return _points(_Volume(_scene(case)), g, n, exclusive=False)
    if op == "shape":
        r = float(_solid(case).rad[0])
        side = 0.4 if case["what"] in ("dist_in", "safety_in") else 1.5
        return [_rand(g, n, -side * r, side * r) + SOLID_TRANS[k] for k in range(3)] + _directions(g, n)
    if op == "batched":
        vols, baskets = _baskets(case)
        out = [torch.empty(n, dtype=F64, device=DEV) for _ in range(6)]
        off = np.concatenate([[0], np.cumsum([c for _, c in baskets])])
        for v in range(len(vols)):
            mine = [(int(off[b]), int(c)) for b, (w, c) in enumerate(baskets) if w == v]
            m = sum(c for _, c in mine)
            if m == 0:
                continue
            T = _points(_Volume(vols[v]), g, m) + _directions(g, m)
            a = 0
            for o, c in mine:
                for k in range(6):
                    out[k][o:o + c] = T[k][a:a + c]
                a += c
        return out
    raise ValueError(op)


def _transport(world, half, g, n):
    """n live tracks after two steps through the tree: fields, node, flag."""
    parts, have = [], 0
    while have < n:
        m = int(1.6 * (n - have)) + 256
        T = [_rand(g, m, -half[k], half[k]) for k in range(3)] + _directions(g, m)
        node = geo.geo_world_locate(world, *T[:3])
        flag = torch.full((m,), -1, dtype=torch.int32, device=DEV)
        for _ in range(2):
            s, node, flag = geo.geo_world_step(world, *T, node, flag)
            live = node >= 0
            T = [T[k] + s * T[3 + k] for k in range(3)] + T[3:]
            T, node, flag = [c[live].contiguous() for c in T], node[live].contiguous(), flag[live].contiguous()
        parts.append(T + [node, flag])
        have += node.numel()
    return [torch.cat([q[k] for q in parts])[:n].contiguous() for k in range(8)]


def prepare(case, seed):
    """The handles and device tensors a user's program holds before the call."""
    op = case["op"]
    if op == "world":
        tree = _world(case)
        world = _build_world(tree)
        half = tree.volumes[tree.root].mother_params[:3]
        return {"case": case, "world": world, "t": _transport(world, half, _generator(seed), case["n"])}
    t = _inputs(case, seed)
    st = {"case": case, "t": t}
    if op == "batched":
        vols, baskets = _baskets(case)
        off = np.concatenate([[0], np.cumsum([c for _, c in baskets])[:-1]])
        handles = [geo.geo_build_volume(s) for s in vols]
        st["batch"] = geo.geo_build_batch(handles, [(v, int(o), c) for (v, c), o in zip(baskets, off)])
    elif op != "shape":
        st["vol"] = geo.geo_build_volume(_scene(case), voxelize=case.get("grid", False))
    if op == "adjoint":
        sc = _scene(case)
        st["p"] = torch.stack(t[:3]).requires_grad_()
        st["d"] = torch.stack(t[3:6]).requires_grad_()
        st["trans"] = _t(sc.trans).requires_grad_()
        st["params"] = _t(np.concatenate([sc.params, sc.mother_params[None, :]])).requires_grad_()
    return st


def run(state):
    case, t = state["case"], state.get("t")
    op = case["op"]
    if op == "step":
        return geo.geo_dist_to_boundary(state["vol"], *t, mode=case["mode"], want_bpoint=case["bpoint"])
    if op == "batched":
        return geo.geo_dist_to_boundary_batched(state["batch"], *t)
    if op == "adjoint":
        leaves = [state[k] for k in ("p", "d", "trans", "params")]
        step, hit = autograd.dist_to_boundary(state["vol"], *leaves)
        return [step.detach(), hit, *torch.autograd.grad(step, leaves, t[6])]
    if op == "contains":
        return geo.geo_contains(state["vol"], *t, mode=case["mode"])
    if op == "safety":
        return geo.geo_safety(state["vol"], *t, mode=case["mode"])
    if op == "world":
        return geo.geo_world_step(state["world"], *t, mode=case["mode"])
    kind, spec = SOLIDS[case["solid"]]
    dist = case["what"].startswith("dist")
    return geo.geo_shape_query(kind, spec, WHAT[case["what"]], *t[:3], *(t[3:] if dist else ()), rot=SOLID_ROT,
                               trans=SOLID_TRANS, want_face=dist)


# FP64 operations (an FMA is two) that one answer needs: the winning solid's
# transform and surface (a quadric: coefficients, square root, division)
_SURFACE_FLOPS = 120.0


def work(case):
    n, op = case["n"], case["op"]
    per = {"step": 60 + (24 if case.get("bpoint") else 0), "batched": 60, "adjoint": 60 + 60 + 48, "contains": 28,
           "safety": 32, "world": 72, "shape": 60 if str(case.get("what", "")).startswith("dist") else 32}[op]
    flops = {"adjoint": 2.5 * _SURFACE_FLOPS, "contains": 10.0, "safety": 40.0}.get(op, _SURFACE_FLOPS)
    return {"bytes": float(per * n), "flops": float(flops * n)}


# --------------------------------------------------------------------------
# exact answers
# --------------------------------------------------------------------------

def _exact_adjoint(case, t):
    """step, hit and the gradients of sum(w * step): the crossing of the
    winning solid that the step ends on, differentiated by torch."""
    sc = _scene(case)
    v = _Volume(sc)
    P, D, w = t[:3], t[3:6], t[6]
    step, hit = v.step(P, D)
    p, d = torch.stack(P).requires_grad_(), torch.stack(D).requires_grad_()
    trans = _t(sc.trans).requires_grad_()
    params = _t(np.concatenate([sc.params, sc.mother_params[None, :]])).requires_grad_()
    total = torch.zeros((), dtype=F64, device=DEV)
    for j in range(-1, v.nd):
        i = (hit == j).nonzero(as_tuple=True)[0]
        if i.numel() == 0:
            continue
        if j < 0:
            x, u, kind, prm = list(p[:, i]), list(d[:, i]), v.mkind, params[-1]
        else:
            W, R = p[:, i] - trans[j][:, None], v.rot[j]
            x, u, kind, prm = list(R.T @ W), list(R.T @ d[:, i]), v.kinds[j], params[j]
        c = torch.stack(torch.broadcast_tensors(*_crossings(kind, list(prm), None, x, u)))
        k = (c.detach() - step[i]).abs().argmin(dim=0)
        total = total + (w[i] * c.gather(0, k[None])[0]).sum()
    return [step, hit, *torch.autograd.grad(total, (p, d, trans, params))]


def _exact_world(case, t):
    tree = _world(case)
    node, flag = t[6], t[7]
    vols = [_Volume(s) for s in tree.volumes]
    # placed volumes breadth first, with their world transforms
    lv, xf = [tree.root], [(np.eye(3), np.zeros(3))]
    k = 0
    while k < len(lv):
        s, (R, o) = tree.volumes[lv[k]], xf[k]
        for j in range(s.n_daughters):
            lv.append(tree.child[lv[k]][j])
            xf.append((R @ s.rot[j].reshape(3, 3), R @ s.trans[j] + o))
        k += 1
    step = torch.full((case["n"],), math.nan, dtype=F64, device=DEV)
    for k in range(len(lv)):
        i = (node == k).nonzero(as_tuple=True)[0]
        if i.numel() == 0:
            continue
        R, o = _t(xf[k][0]), _t(xf[k][1])
        W, E = [t[c][i] - o[c] for c in range(3)], [t[3 + c][i] for c in range(3)]
        x = [R[0, c] * W[0] + R[1, c] * W[1] + R[2, c] * W[2] for c in range(3)]
        u = [R[0, c] * E[0] + R[1, c] * E[1] + R[2, c] * E[2] for c in range(3)]
        step[i] = vols[lv[k]].step(x, u, skip=flag[i], entered=flag[i] == -2)[0]
    return [step, None, None]


def _exact_shape(case, t):
    one = _solid(case)
    kind, planes, p = one.kinds[0], one.groups[0][2], list(one.prm[0])
    W, R = torch.stack([t[k] - one.trans[0, k] for k in range(3)]), one.rot[0]
    x = [R[0, c] * W[0] + R[1, c] * W[1] + R[2, c] * W[2] for c in range(3)]
    u = [R[0, c] * t[3] + R[1, c] * t[4] + R[2, c] * t[5] for c in range(3)]
    what = case["what"]
    if what == "contains":
        return _inside(kind, p, planes, x).to(F64)
    if what.startswith("safety"):
        return _safety(kind, p, planes, x, what == "safety_in")
    if what == "dist_out":
        return [_along(kind, p, planes, x, u, True), None]
    return [torch.where(_inside(kind, p, planes, x), _along(kind, p, planes, x, u, False), 0.0), None]


def exact(case, seed):
    op = case["op"]
    if op == "world":
        return _exact_world(case, prepare(case, seed)["t"])
    t = _inputs(case, seed)
    if op == "adjoint":
        return _exact_adjoint(case, t)
    if op == "shape":
        return _exact_shape(case, t)
    if op == "batched":
        vols, baskets = _baskets(case)
        step = torch.empty(case["n"], dtype=F64, device=DEV)
        hit = torch.empty(case["n"], dtype=torch.int32, device=DEV)
        off = np.concatenate([[0], np.cumsum([c for _, c in baskets])])
        for v in range(len(vols)):
            mine = [torch.arange(int(off[b]), int(off[b + 1]), device=DEV) for b, (w, _) in enumerate(baskets) if w == v]
            if mine:
                i = torch.cat(mine)
                T = [c[i] for c in t]
                step[i], hit[i] = _Volume(vols[v]).step(T[:3], T[3:])
        return [step, hit]
    v = _Volume(_scene(case))
    if op == "contains":
        return v.contains(t)
    if op == "safety":
        return None if case["mode"] == geo.GEO_SAFETY_ESTIMATE else v.safety(t)
    step, hit = v.step(t[:3], t[3:])
    out = [step, hit]
    if case["bpoint"]:
        out.append(torch.stack([t[k] + step * t[3 + k] for k in range(3)]))
    return out
