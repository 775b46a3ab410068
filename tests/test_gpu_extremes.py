"""Inputs at the ends of their ranges: both modes and every kernel give the
plain FP64 routines' bits there too."""
import numpy as np
import pytest

from paper_1312_0816_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EYE = np.eye(3).reshape(9)


@pytest.fixture(scope="module")
def g():
    import paper_1312_0816_gb300 as pkg

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.load()
    return pkg


def cuda(*arrays):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]


def same(a, b):
    return torch.equal(a[0].view(torch.int64), b[0].view(torch.int64)) and all(torch.equal(x, y) for x, y in zip(a[1:], b[1:]))


@pytest.mark.parametrize("extent", [1e3, 1e4, 1e5, 1e6, 1e7])
@pytest.mark.parametrize("rotated", [False, True])
def test_small_solids_in_a_large_mother(g, extent, rotated):
    """Tracks from far away that graze small solids, within the rounding of the
    quadrics' crossings and beyond: the FP64 culls (annuli and spheres, lists
    and the walk of a one-cell grid) pass every line that the whole routine
    accepts, so the modes and the kernels agree."""
    rng = np.random.default_rng(int(extent) + rotated)
    n = 200003
    kinds = [(scenes.TUBE, (0.0, 5.0, 100.0)), (scenes.CONE, (100.0, 1.0, 4.0, 2.0, 6.0)), (scenes.TUBE, (4.0, 5.0, 50.0)),
             (scenes.CONE, (0.5, 2.0, 4.0, 3.0, 9.0)), (scenes.TUBE, (0.0, 0.1, 80.0)), (scenes.TUBE, (0.0, 5.0, 0.05))]
    rows = [(*kinds[k % 6], scenes.haar_rotation(rng) if rotated else EYE,
             (0.0, 0.0, 0.0) if k % 4 == 0 else (30.0 * k - 500.0, 3.0 * k, 0.0)) for k in range(36)]
    sc = scenes._scene("far", scenes.BOX, (extent,) * 3, rows)
    flat, walk = g.geo_build_volume(sc), g.geo_build_volume(sc, voxelize=True, grid=(1, 1, 1))
    j = rng.integers(0, len(rows), n)
    prm, cone = sc.params[j], sc.kinds[j] == scenes.CONE
    half = np.where(cone, prm[:, 0], prm[:, 2])
    z = rng.uniform(-1.01, 1.01, n) * half
    slope = np.where(cone, (prm[:, 4] - prm[:, 2]) / (2.0 * half), 0.0)
    radius = np.where(cone, 0.5 * (prm[:, 2] + prm[:, 4]), prm[:, 1]) + slope * z
    radius = np.where(rng.random(n) < 0.2, np.where(cone, 1.5, np.maximum(prm[:, 0], 0.05)), radius)
    b = radius * (1.0 + 10.0 ** rng.uniform(-14.0, -2.0, n) * rng.choice([-1.0, 1.0], n))
    ph = rng.uniform(0.0, 2.0 * np.pi, n)
    u = np.stack([np.cos(ph), np.sin(ph), slope * 0.0 + rng.normal(0.0, 0.3, n) * rng.integers(0, 2, n)])
    u /= np.linalg.norm(u, axis=0)
    foot = np.stack([-b * np.sin(ph), b * np.cos(ph), z])
    local = foot - u * rng.uniform(0.05, 0.65, n) * (extent - 600.0)
    R = sc.rot[j].reshape(n, 3, 3)
    p = np.einsum("nab,bn->an", R, local) + sc.trans[j].T
    t = cuda(*p, *np.einsum("nab,bn->an", R, u))
    f0 = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
    assert int((f0[1] >= 0).sum()) > n // 4
    assert same(f0, g.geo_dist_to_boundary(walk, *t, mode=g.GEO_FP64))
    for v in (flat, walk):
        assert same(f0, g.geo_dist_to_boundary(v, *t, mode=g.GEO_FP32_REFINE))
    # the step of a track and the whole routine of the solid it enters
    for k in range(6):
        i = torch.nonzero(f0[1] == k).flatten()
        kind, q = rows[k][0], rows[k][1]
        own = g.geo_shape_query(kind, q, g.GEO_Q_DIST_OUT, *[x[i].contiguous() for x in t], rot=rows[k][2], trans=rows[k][3])
        assert torch.equal(own.view(torch.int64), f0[0][i].view(torch.int64))


@pytest.mark.parametrize("scene", ["shells", "thin"])
@pytest.mark.parametrize("length", [1.0, 1e-6, 1e-9, 1e-10, 1e-11, 1e-12, 1e-13, 1e-14, 1.2e-15])
def test_short_directions(g, scene, length):
    """Directions from units down to where their squares leave the normal FP32
    range, inclined to the solids' axis by anything from 1e-6 on."""
    rng = np.random.default_rng(5)
    n = 60007
    if scene == "shells":
        cone = (5.0, 1.0, 12.0, 2.0, 20.0)
        rows = [(scenes.TUBE, (0.0, 10.0, 5.0), EYE, (0.0, 0.0, 40.0 * k)) for k in range(-4, 5)]
        rows += [(scenes.CONE, cone, EYE, (60.0, 0.0, 40.0 * k)) for k in range(-8, 9)]
        rows += [(scenes.TUBE, (3.0, 10.0, 5.0), EYE, (-60.0, 0.0, 40.0 * k)) for k in range(-8, 9)]
        sc = scenes._scene("shells", scenes.BOX, (400.0,) * 3, rows)
        p = np.stack([rng.choice([0.0, 60.0, -60.0], n) + rng.uniform(-9.0, 9.0, n), rng.uniform(-9.0, 9.0, n),
                      rng.uniform(-390.0, 390.0, n)])
    else:
        rows = [(scenes.TUBE, (2e-3, 4e-3, 1.0), EYE, (0.0, 0.0, 2.0)),
                (scenes.CONE, (1.0, 1e-3, 2e-3, 3e-3, 5e-3), EYE, (0.0, 0.0, -2.0))] * 17
        sc = scenes._scene("thin", scenes.TUBE, (0.0, 1e-2, 5.0), rows)
        p = np.stack([rng.uniform(-6e-3, 6e-3, n), rng.uniform(-6e-3, 6e-3, n), rng.uniform(-4.9, 4.9, n)])
    s, ph = 10.0 ** rng.uniform(-6.0, -0.1, n), rng.uniform(0.0, 2.0 * np.pi, n)
    t = cuda(*p, *(np.stack([s * np.cos(ph), s * np.sin(ph), rng.choice([-1.0, 1.0], n)]) * length))
    flat, grid = g.geo_build_volume(sc), g.geo_build_volume(sc, voxelize=True)
    ref = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
    assert same(ref, g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP32_REFINE))
    batch = g.geo_build_batch([flat], [(0, 0, n)])
    assert same(ref, g.geo_dist_to_boundary_batched(batch, *t))
    few = [x[:1000].contiguous() for x in t]   # the small-basket kernel
    assert same([x[:1000] for x in ref], g.geo_dist_to_boundary(flat, *few, mode=g.GEO_FP32_REFINE))
    # the tree: the volume in a hall, its daughters leaves
    leaves = [g.geo_build_volume(scenes.leaf(int(k), q)) for k, q in zip(sc.kinds, sc.params)]
    hall = g.geo_build_volume(scenes._scene("hall", scenes.BOX, (500.0,) * 3, [(sc.mother_kind, sc.mother_params, EYE, (0, 0, 0))]))
    m = len(leaves)
    world = g.geo_build_world(leaves + [flat, hall], [[] for _ in leaves] + [list(range(m)), [m]], m + 1)
    node = torch.full((n,), 1, dtype=torch.int32, device="cuda")
    a = g.geo_world_step(world, *t, node, mode=g.GEO_FP64)
    assert same(a, g.geo_world_step(world, *t, node, mode=g.GEO_FP32_REFINE))


@pytest.mark.parametrize("length", [1.0, 1e-9, 1e-11, 1e-13, 1.2e-15])
@pytest.mark.parametrize("kind,prm", [(scenes.TUBE, (3.0, 10.0, 5.0)), (scenes.CONE, (5.0, 1.0, 12.0, 2.0, 20.0)),
                                      (scenes.TUBE, (0.0, 1e-2, 5.0)), (scenes.BOX, (3.0, 10.0, 5.0))])
def test_short_directions_of_one_solid(g, kind, prm, length):
    """The list kernel (from 98304 tracks on) against the whole routine's."""
    rng = np.random.default_rng(6)
    n, m = 98304, 90000
    s, ph = 10.0 ** rng.uniform(-6.0, -0.1, n), rng.uniform(0.0, 2.0 * np.pi, n)
    size = 1.2 * np.array({scenes.BOX: prm[:3], scenes.TUBE: (prm[1], prm[1], prm[-1])}.get(kind, (20.0, 20.0, 5.0)))
    p = rng.uniform(-1.0, 1.0, (3, n)) * size[:, None]
    p[2] += 10.0 * rng.integers(-1, 2, n)
    t = cuda(*p, *(np.stack([s * np.cos(ph), s * np.sin(ph), rng.choice([-1.0, 1.0], n)]) * length))
    for what in (g.GEO_Q_DIST_OUT, g.GEO_Q_DIST_IN):
        a = g.geo_shape_query(kind, prm, what, *t, want_face=True)
        b = g.geo_shape_query(kind, prm, what, *[x[:m].contiguous() for x in t], want_face=True)
        assert same([x[:m] for x in a], b)


HOLED = {"cone": (scenes.CONE, (100.0, 30.0, 90.0, 50.0, 120.0)), "tube": (scenes.TUBE, (40.0, 90.0, 100.0)),
         "tubs": (scenes.TUBS, (40.0, 90.0, 100.0, 0.2, 5.0)),
         "pcon": (scenes.PCON, scenes.Pcon((-100.0, -20.0, 20.0, 100.0), (20.0, 38.0, 42.0, 30.0), (90.0, 95.0, 95.0, 90.0)))}


@pytest.mark.parametrize("copies", [1, 3])   # 12 daughters, 36
@pytest.mark.parametrize("mother", sorted(HOLED))
def test_starts_on_the_surface_of_the_mothers_hole(g, mother, copies):
    """Tracks that start within a rounding of the hole of their mother and move
    into it: FP64 may pass over the crossing at the start, and the daughters
    beyond the hole then decide the step."""
    rng = np.random.default_rng(copies)
    n = 200003
    kind, prm = HOLED[mother]
    a = 2.0 * np.pi / 12 * np.arange(12)
    rows = [(scenes.BOX, (6.0, 6.0, 20.0), scenes._rot_z(p), (70.0 * np.cos(p), 70.0 * np.sin(p), 0.0)) for p in a] * copies
    sc = scenes._scene("holed", kind, prm, rows)
    ph = rng.uniform(0.0, 2.0 * np.pi, n)
    z = rng.uniform(-90.0, 90.0, n) if mother == "pcon" else rng.uniform(-30.0, 30.0, n)
    if mother == "cone":
        ri = 40.0 + 0.1 * z
    elif mother == "pcon":
        zp, rn, _ = sc.planes_of(sc.mother_params)
        ri = np.interp(z, zp, rn)
    else:
        ri = np.full(n, 40.0)
    r = ri * (1.0 + rng.integers(-2, 3, n) * 2.0 ** -53)
    d = -np.stack([np.cos(ph + rng.normal(0.0, 0.3, n)), np.sin(ph + rng.normal(0.0, 0.3, n)), rng.normal(0.0, 0.1, n)])
    t = cuda(r * np.cos(ph), r * np.sin(ph), z, *d)
    flat = g.geo_build_volume(sc)
    ref = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
    assert int((ref[1] > -2).sum()) > n // 4
    assert same(ref, g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP32_REFINE))
    grid = g.geo_build_volume(sc, voxelize=True)
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary_batched(g.geo_build_batch([flat], [(0, 0, n)]), *t))
    few = [x[:1000].contiguous() for x in t]
    assert same([x[:1000] for x in ref], g.geo_dist_to_boundary(flat, *few, mode=g.GEO_FP32_REFINE))
    # the tree: tracks in the volume, or just entered and scattered back
    seg = (scenes.TUBS, (1.0, 2.0, 3.0, 0.0, 1.0))
    for other in ([], [(*seg, EYE, (300.0, 0.0, 0.0))]):   # with a segment: the tiled kernel
        hall = scenes._scene("hall", scenes.BOX, (500.0,) * 3, [(kind, prm, EYE, (0.0, 0.0, 0.0))] + other)
        vols = [g.geo_build_volume(s) for s in (scenes.leaf(scenes.BOX, (6.0, 6.0, 20.0)), sc, hall)]
        child = [[], [0] * len(rows), [1]]
        if other:
            vols.append(g.geo_build_volume(scenes.leaf(*seg)))
            child = child[:2] + [[1, 3], []]
        world = g.geo_build_world(vols, child, 2)
        node = torch.ones(n, dtype=torch.int32, device="cuda")
        for f in (-1, -2):
            flag = torch.full((n,), f, dtype=torch.int32, device="cuda")
            assert same(g.geo_world_step(world, *t, node, flag, mode=g.GEO_FP64),
                        g.geo_world_step(world, *t, node, flag, mode=g.GEO_FP32_REFINE))


@pytest.mark.parametrize("kind,prm", [(scenes.BOX, (3.0, 20.0, 11.0)), (scenes.TUBE, (0.0, 9.0, 14.0)),
                                      (scenes.TUBE, (8.9, 9.0, 4.0)), (scenes.CONE, (5.0, 1.0, 30.0, 20.0, 21.0)),
                                      (scenes.CONE, (30.0, 2.0, 4.0, 9.0, 9.0)), (scenes.CONE, (0.5, 2.0, 4.0, 30.0, 40.0))])
@pytest.mark.parametrize("reach", [2.0, 9.0, 30.0, 1e3, 1e6, 1e12, 1e17, 1e200])
def test_one_solid_from_afar(g, kind, prm, reach):
    """Points up to `reach` times the solid's size away, half of them on its
    surface or on lines that graze it, through the list kernels (from 98304 points
    on; Contains always) against the whole routines'."""
    rng = np.random.default_rng(int(np.log10(reach) * 10.0))
    n, m = 98304, 90000
    R, shift = scenes.haar_rotation(rng), np.array([7.0, -3.0, 5.0])
    size = max(prm)
    # points on the faces, and directions along them or anywhere
    if kind == scenes.BOX:
        q = rng.uniform(-1.0, 1.0, (n, 3))
        q[np.arange(n), rng.integers(0, 3, n)] = rng.choice([-1.0, 1.0], n)
        q *= np.array(prm)
    else:
        ends = (prm[0], prm[1], prm[0], prm[1], prm[2]) if kind == scenes.TUBE else (*prm[1:], prm[0])
        f, ph = rng.uniform(0.0, 1.0, n), rng.uniform(0.0, 2.0 * np.pi, n)
        f = np.where(rng.random(n) < 0.2, rng.integers(0, 2, n), f)
        lo, hi = ends[0] + f * (ends[2] - ends[0]), ends[1] + f * (ends[3] - ends[1])
        r = np.where(rng.random(n) < 0.5, hi, np.where(rng.random(n) < 0.5, lo, rng.uniform(0.0, 1.0, n) * (hi - lo) + lo))
        q = np.stack([r * np.cos(ph), r * np.sin(ph), (2.0 * f - 1.0) * ends[4]], axis=1)
    d = np.stack(scenes.isotropic(rng, n), axis=1)
    graze = rng.random(n) < 0.3
    d[graze, 2] = 0.0 if kind == scenes.TUBE else d[graze, 2]
    radial = np.stack([-q[:, 1], q[:, 0], np.zeros(n)], axis=1) / np.maximum(np.hypot(q[:, 0], q[:, 1]), 1e-300)[:, None]
    d[graze] = radial[graze] + 1e-3 * rng.normal(0.0, 1.0, (int(graze.sum()), 3)) * rng.integers(0, 2, (int(graze.sum()), 1))
    away = size * reach ** rng.uniform(0.0, 1.0, (n, 1)) * rng.choice([0.0, 1.0, 1.0, 1.0], (n, 1)) * rng.choice([-1.0, 1.0], (n, 1))
    p = q - d * away
    anywhere = rng.random(n) < 0.4
    p[anywhere] = rng.normal(0.0, 1.0, (int(anywhere.sum()), 3)) * size * reach ** rng.uniform(0.0, 1.0, (int(anywhere.sum()), 1))
    A = R.reshape(3, 3)
    t = cuda(*(p @ A.T + shift).T, *(d @ A.T).T)
    for what in (g.GEO_Q_DIST_OUT, g.GEO_Q_DIST_IN, g.GEO_Q_SAFETY_OUT, g.GEO_Q_SAFETY_IN):
        dist = what in (g.GEO_Q_DIST_OUT, g.GEO_Q_DIST_IN)
        a = g.geo_shape_query(kind, prm, what, *t[:6 if dist else 3], rot=R, trans=shift, want_face=True)
        b = g.geo_shape_query(kind, prm, what, *[x[:m].contiguous() for x in t[:6 if dist else 3]], rot=R, trans=shift,
                              want_face=True)
        assert same([x[:m] for x in a], b)
        if what == g.GEO_Q_DIST_IN:   # the whole routine's face tells whether it holds the point
            inside = g.geo_shape_query(kind, prm, g.GEO_Q_CONTAINS, *t[:3], rot=R, trans=shift) == 1.0
            assert torch.equal(inside[:m] & ~torch.isnan(b[0]), b[1] >= 0)   # (NaN: no direction, on the axis)


MOTHERS = {**HOLED, "box": (scenes.BOX, (90.0, 95.0, 100.0)), "rod": (scenes.TUBE, (0.0, 90.0, 100.0)),
           "plug": (scenes.CONE, (100.0, 0.0, 90.0, 0.0, 120.0))}


@pytest.mark.parametrize("daughters", ["few", "many", "overlapping"])
@pytest.mark.parametrize("mother", sorted(MOTHERS))
def test_starts_on_the_mothers_surface(g, mother, daughters):
    """Tracks that start on a face of their mother, a rounding or up to 1e-3 of
    her size inside, in any direction, along the face or nearly so: the mother's
    exit is bounded there as for a track that has just entered."""
    rng = np.random.default_rng(len(mother) * 10 + len(daughters))
    n = 200003
    kind, prm = MOTHERS[mother]
    count = {"few": 12, "many": 60, "overlapping": 40}[daughters]
    rows = []
    for k in range(count):
        a, r = 2.0 * np.pi * k / min(count, 12), rng.uniform(60.0, 68.0)
        size = rng.uniform(2.0, 8.0 if daughters != "overlapping" else 12.0, 3)   # inside the outer surface
        at = (r * np.cos(a), r * np.sin(a), rng.uniform(-79.0, 79.0))
        solid = [(scenes.BOX, size), (scenes.TUBE, (0.3 * size[0], size[0], size[1])),
                 (scenes.CONE, (size[2], 0.1, size[0], 0.2, size[1]))][k % 3]
        rows.append((*solid, scenes.haar_rotation(rng) if k % 2 else EYE, at))
    sc = scenes._scene("skin", kind, prm, rows)
    face, ph = rng.integers(0, 3, n), rng.uniform(0.0, 2.0 * np.pi, n)
    z = np.where(face == 0, 100.0 * rng.choice([-1.0, 1.0], n), rng.uniform(-100.0, 100.0, n))
    if kind == scenes.BOX:
        p = rng.uniform(-1.0, 1.0, (3, n)) * np.array(prm)[:, None]
        p[face, np.arange(n)] = np.array(prm)[face] * rng.choice([-1.0, 1.0], n)
        normal = np.zeros((3, n))
        normal[face, np.arange(n)] = np.sign(p[face, np.arange(n)])
    else:
        if kind == scenes.PCON:
            zp, rn, rx = sc.planes_of(sc.mother_params)
        else:
            zp = np.array([-100.0, 100.0])
            rn, rx = ((np.array([prm[1], prm[3]]), np.array([prm[2], prm[4]])) if kind == scenes.CONE
                      else (np.full(2, prm[0]), np.full(2, prm[1])))
        ro, ri = np.interp(z, zp, rx), np.interp(z, zp, rn)
        r = np.where(face == 0, ri + rng.uniform(0.0, 1.0, n) * (ro - ri), np.where(face == 1, ro, ri))
        p = np.stack([r * np.cos(ph), r * np.sin(ph), z])
        side = np.where(face == 1, 1.0, -1.0)
        normal = np.where(face == 0, np.stack([0.0 * z, 0.0 * z, np.sign(z)]), np.stack([side * np.cos(ph), side * np.sin(ph), 0.0 * z]))
    depth = rng.choice([0.0, 1e-15, 1e-13, 1e-9, 1e-6, 1e-5, 1e-4, 1e-3], n) * 100.0
    p = p - normal * depth
    d = np.stack(scenes.isotropic(rng, n))
    flat_along = rng.random(n) < 0.3   # along the face, but for a little
    along = d - normal * (normal * d).sum(axis=0)
    d = np.where(flat_along, along + normal * rng.choice([0.0, 1e-12, 1e-7, 1e-4], n) * rng.choice([-1.0, 1.0], n), d)
    t = cuda(*p, *d)
    flat, grid = g.geo_build_volume(sc), g.geo_build_volume(sc, voxelize=True)
    ref = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
    assert int((ref[1] > -2).sum()) > n // 4
    assert same(ref, g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP64))
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary_batched(g.geo_build_batch([flat], [(0, 0, n)]), *t))
    assert same(ref, g.geo_dist_to_boundary_batched(g.geo_build_batch([grid], [(0, 0, n)]), *t))
    few = [x[:1000].contiguous() for x in t]
    assert same([x[:1000] for x in ref], g.geo_dist_to_boundary(flat, *few, mode=g.GEO_FP32_REFINE))


@pytest.mark.parametrize("cells", [(0, 0, 0), (7, 3, 40)])
@pytest.mark.parametrize("half", [(90.0, 95.0, 100.0), (0.1, 70.0, 1.3)])
def test_starts_along_a_wall_of_the_grid(g, half, cells):
    """Tracks a rounding (FP32's or FP64's) inside a wall of the mother's box and
    of the grid, moving along it and hardly towards it, with daughters flush with
    the wall ahead."""
    rng = np.random.default_rng(int(half[1]))
    n = 200003
    half = np.array(half)
    rows = []
    for k in range(3):
        for side in (-1.0, 1.0):
            for _ in range(10):
                size = half * rng.uniform(0.03, 0.1, 3)
                size[k] = half[k] / 16
                at = rng.uniform(-0.85, 0.85, 3) * half
                at[k] = side * (half[k] - size[k])
                rows.append((scenes.BOX, size, EYE, at))
    sc = scenes._scene("flush", scenes.BOX, half, rows)
    face, side = rng.integers(0, 3, n), rng.choice([-1.0, 1.0], n)
    i = np.arange(n)
    p = rng.uniform(-1.0, 1.0, (3, n)) * half[:, None]
    p[face, i] = side * half[face] * (1.0 - rng.choice([0.0, 1e-15, 1e-14, 1e-12, 1e-9, 1e-8, 1e-7], n))
    d = np.stack(scenes.isotropic(rng, n))
    d[face, i] = side * rng.choice([0.0, 1e-20, 1e-18, 1e-16, 1e-14, 1e-12, 1e-10, 1e-8], n)
    t = cuda(*p, *d)
    flat, grid = g.geo_build_volume(sc), g.geo_build_volume(sc, voxelize=True, grid=cells)
    ref = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
    assert int((ref[1] >= 0).sum()) > n // 20
    assert same(ref, g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP64))
    assert same(ref, g.geo_dist_to_boundary(grid, *t, mode=g.GEO_FP32_REFINE))
    assert same([x[:60000] for x in ref], g.geo_dist_to_boundary(grid, *[x[:60000].contiguous() for x in t]))
    assert same(ref, g.geo_dist_to_boundary_batched(g.geo_build_batch([grid], [(0, 0, n)]), *t))


@pytest.mark.parametrize("scene", ["toy8", "toy40", "grid512"])
def test_starts_on_the_daughters_surfaces(g, scene):
    """Tracks that start where an earlier step ended, or a little beside it, in any
    direction: FP32 is certain of nothing there, and whole solids are evaluated.
    The reference walks a grid of one cell with the shapes' own functions."""
    sc = scenes.SCENES[scene]()
    rng = np.random.default_rng(9)
    n = 260011
    tr = scenes.sample_tracks(sc, n, 9)
    t = cuda(*tr.fields())
    flat, walk, grid = (g.geo_build_volume(sc, **o) for o in ({}, {"voxelize": True, "grid": (1, 1, 1)}, {"voxelize": True}))
    s, h = g.geo_dist_to_boundary(walk, *t, mode=g.GEO_FP64)
    i = torch.nonzero(h >= 0).flatten()
    i = i[torch.from_numpy(rng.integers(0, i.numel(), n)).cuda()]
    s = s[i] + torch.from_numpy(rng.choice([0.0, 0.0, -1e-12, 1e-12, -1e-9, 1e-9, -1e-4, 1e-4], n)).cuda()
    p = [(t[k][i] + s * t[3 + k][i]).contiguous() for k in range(3)]
    q = p + cuda(*np.stack(scenes.isotropic(rng, n)))
    ref = g.geo_dist_to_boundary(walk, *q, mode=g.GEO_FP64)
    for v in (flat, grid):
        for m in (n, 60011):
            part = [x[:m].contiguous() for x in q]
            assert same([x[:m] for x in ref], g.geo_dist_to_boundary(v, *part, mode=g.GEO_FP32_REFINE))
    assert same(ref, g.geo_dist_to_boundary(flat, *q, mode=g.GEO_FP64))
    for v in (flat, grid):
        assert same(ref, g.geo_dist_to_boundary_batched(g.geo_build_batch([v], [(0, 0, n)]), *q))
    for m in (n, 60011, 1009):
        part = [x[:m].contiguous() for x in p]
        assert torch.equal(g.geo_contains(flat, *part, mode=g.GEO_FP64), g.geo_contains(flat, *part))
        a, b = g.geo_safety(flat, *part, mode=g.GEO_FP64), g.geo_safety(flat, *part)
        assert torch.equal(a.view(torch.int64), b.view(torch.int64))


@pytest.mark.parametrize("n", [33, 5003, 170003])
@pytest.mark.parametrize("daughters", [31, 32, 40, 70])
def test_safety_of_points_with_many_nearest_solids(g, daughters, n):
    """Points on and near the axis of a ring of equal solids, and anywhere: more
    than two candidates are too close to tell apart in FP32."""
    rng = np.random.default_rng(daughters + n)
    rows = []
    for k in range(daughters):
        a = 2.0 * np.pi * k / daughters
        at = (60.0 * np.cos(a), 60.0 * np.sin(a), 0.0)
        solid = [(scenes.BOX, (1.0, 1.5, 9.0)), (scenes.TUBE, (0.4, 1.0, 9.0)), (scenes.CONE, (9.0, 0.2, 1.0, 0.3, 1.0))][k % 3]
        rows.append((*solid, scenes._rot_z(a), at))
    sc = scenes._scene("ring", scenes.TUBE, (0.0, 200.0, 150.0), rows)
    vol = g.geo_build_volume(sc)
    p = rng.normal(0.0, 1.0, (3, n)) * rng.choice([0.0, 1e-12, 1e-7, 1e-5, 1e-3, 50.0], n)
    p[2] += rng.uniform(-8.0, 8.0, n) * rng.integers(0, 2, n)
    t = cuda(*p)
    a, b = g.geo_safety(vol, *t, mode=g.GEO_FP64), g.geo_safety(vol, *t)
    assert torch.equal(a.view(torch.int64), b.view(torch.int64))
