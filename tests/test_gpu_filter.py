"""The filter's tables and the surfaces it is certain of: volumes whose numbers
of unrotated quadrics, rotated quadrics and boxes sit at the edges of the
32-entry chunks and of the pairs, staged in shared memory or read from global
memory, for one basket and for a batch.  The answers are the plain FP64
kernel's bits (GEO_FP64 evaluates every solid whole, without the filter)."""
import numpy as np
import pytest

from paper_1312_0816_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_1312_0816_gb300 as pkg

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.load()
    return pkg


def filter_scene(n1, n2, n3, mother, seed, apex=False):
    """n1 unrotated tubes and cones (nested shells about two axes: shells of no
    thickness, holes far narrower than the filter's inflation), n2 rotated
    ones (apex: cones ending in an apex too, whose volumes take other
    kernels), n3 boxes; they may overlap."""
    rng = np.random.default_rng(seed)
    eye = np.eye(3).reshape(9)
    rows = []
    for k in range(n1):
        axis = ((0.0, 0.0), (0.0, 0.0), (60.0, -40.0))[k % 3]
        r = 10.0 + 300.0 * k / max(n1, 1)
        t = (axis[0], axis[1], rng.uniform(-200.0, 200.0))
        if k % 4 == 1:
            r1, r2 = r, r + rng.uniform(-8.0, 30.0)
            rows.append((scenes.CONE, (rng.uniform(5.0, 150.0), r1 * 0.7, r1, r2 * 0.6, r2), eye, t))
        else:
            rmin = (r, r * 0.9, 1e-6, 0.0)[k % 7 % 4]
            rows.append((scenes.TUBE, (rmin, r, rng.uniform(5.0, 300.0)), eye, t))
    for k in range(n2):
        t = rng.uniform(-350.0, 350.0, 3)
        if k % 2:
            rows.append((scenes.CONE, (rng.uniform(5.0, 40.0), 0.0 if apex else 1.0, 0.0 if apex and k % 6 == 1 else 10.0, 2.0, 25.0),
                         scenes.haar_rotation(rng), t))
        else:
            rows.append((scenes.TUBE, (0.0 if k % 4 else 6.0, rng.uniform(8.0, 30.0), rng.uniform(5.0, 40.0)),
                         scenes.haar_rotation(rng), t))
    for k in range(n3):
        rows.append((scenes.BOX, rng.uniform(3.0, 40.0, 3), eye if k % 3 == 0 else scenes.haar_rotation(rng),
                     rng.uniform(-350.0, 350.0, 3)))
    order = rng.permutation(len(rows))
    mk, mp = (scenes.BOX, (400.0, 400.0, 400.0)) if mother == "box" else (scenes.TUBE, (0.0, 420.0, 400.0))
    return scenes._scene(f"filter{n1}_{n2}_{n3}", mk, mp, [rows[i] for i in order])


def tracks(sc, n, seed):
    """Points in the mother (inside daughters and outside the mother too), isotropic
    directions; some along an axis, some in a coordinate plane, some of
    other lengths."""
    rng = np.random.default_rng(seed)
    p = rng.uniform(-405.0, 405.0, (3, n))
    d = np.stack(scenes.isotropic(rng, n))
    m = n // 16
    for k in range(3):
        d[k, k * m:(k + 1) * m] = 0.0                       # in a coordinate plane
        d[:, (3 + k) * m:(4 + k) * m] = 0.0
        d[k, (3 + k) * m:(4 + k) * m] = rng.choice([-1.0, 1.0], m)   # along an axis
    d[:, 7 * m:8 * m] *= 1e-3
    d[:2, 8 * m:9 * m] *= 1e-7                              # nearly along z
    d[2, 9 * m:10 * m] *= 1e-7                              # nearly across it
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p, *d)]


COUNTS = [(0, 0, 1), (1, 0, 0), (1, 1, 1), (2, 1, 0), (31, 2, 5), (32, 0, 0), (33, 0, 1), (34, 31, 1), (1, 32, 32),
          (2, 65, 33), (40, 40, 19), (0, 150, 130), (10, 50, 32)]


@pytest.mark.parametrize("mother,apex", [("box", False), ("tube", False), ("box", True)])
@pytest.mark.parametrize("counts", COUNTS)
def test_filter_equals_fp64_bitwise(g, counts, mother, apex):
    sc = filter_scene(*counts, mother, seed=sum(counts) + 7, apex=apex)
    vol = g.geo_build_volume(sc)
    for n in (257, 70001):   # n = 257: the small-basket kernels; 70001: the direct or the pipelined one
        t = tracks(sc, n, n)
        s0, h0 = g.geo_dist_to_boundary(vol, *t, mode=g.GEO_FP64)
        s1, h1 = g.geo_dist_to_boundary(vol, *t, mode=g.GEO_FP32_REFINE)
        assert torch.equal(h0, h1)
        assert torch.equal(s0.view(torch.int64), s1.view(torch.int64))
    assert len(torch.unique(h1)) > 2
    assert g.geo_check_device_status(vol) == 0


@pytest.mark.parametrize("n", [60013, 600011, 1200007])
@pytest.mark.parametrize("which", [(1, 4, 10), (0, 11, 9, 10)])
def test_batched_filter_equals_fp64_bitwise(g, which, n):
    """Small and large volumes, in baskets from 17 tracks to a third of the
    batch; sizes at which a warp takes 32, 64 and 128 tracks of a tile at a time."""
    vols = [g.geo_build_volume(filter_scene(*COUNTS[w], "box", seed=100 + w)) for w in which]
    t = tracks(None, n, 5)
    cuts = [0, 17, 400, n // 3, n // 3 + 384, 3 * n // 4, n]
    rows = [(k % len(vols), a, b - a) for k, (a, b) in enumerate(zip(cuts, cuts[1:]))]
    for tile in (384, 256):
        batch = g.geo_build_batch(vols, rows, tile_tracks=tile)
        s, h = g.geo_dist_to_boundary_batched(batch, *t)
        for v, a, c in rows:
            s0, h0 = g.geo_dist_to_boundary(vols[v], *[x[a:a + c].contiguous() for x in t], mode=g.GEO_FP64)
            assert torch.equal(h[a:a + c], h0)
            assert torch.equal(s[a:a + c].view(torch.int64), s0.view(torch.int64))
    for v in vols:
        assert g.geo_check_device_status(v) == 0


@pytest.mark.parametrize("grid", [(0, 0, 0), (1, 1, 1), (7, 3, 40)])
@pytest.mark.parametrize("counts", [(1, 1, 1), (34, 31, 1), (0, 150, 130)])
def test_grid_equals_fp64_bitwise(g, counts, grid):
    """The grid's walk with one thread per track (up to 1.25 waves of tracks), and
    with a warp's tracks sorted for FP64, over the staged short form (beyond)."""
    sc = filter_scene(*counts, "box", seed=sum(counts) + 7)
    vol = g.geo_build_volume(sc, voxelize=True, grid=grid)
    wave = 1024 * torch.cuda.get_device_properties(0).multi_processor_count
    for n in (30011, wave * 5 // 4 - 1, wave * 5 // 4, wave * 4 + 333):
        t = tracks(sc, n, n)
        s0, h0 = g.geo_dist_to_boundary(vol, *t, mode=g.GEO_FP64)
        s1, h1 = g.geo_dist_to_boundary(vol, *t, mode=g.GEO_FP32_REFINE)
        assert torch.equal(h0, h1)
        assert torch.equal(s0.view(torch.int64), s1.view(torch.int64))
    # host arrays in place: one thread per track whatever the size
    host = [x.cpu().pin_memory() for x in t]
    s2, h2 = g.geo_dist_to_boundary_host(vol, *host, mode=g.GEO_FP32_REFINE)
    assert torch.equal(h2, h0.cpu()) and torch.equal(s2.view(torch.int64), s0.cpu().view(torch.int64))
    assert g.geo_check_device_status(vol) == 0


@pytest.mark.parametrize("mother,apex", [("box", False), ("tube", False), ("box", True)])
@pytest.mark.parametrize("counts", COUNTS)
def test_fp64_lists_equal_the_single_cell_walk(g, counts, mother, apex):
    """The FP64 step's culls and lists per lane against a grid of one cell, whose
    walk looks at every daughter with the shapes' own functions."""
    sc = filter_scene(*counts, mother, seed=sum(counts) + 7, apex=apex)
    flat, walk = g.geo_build_volume(sc), g.geo_build_volume(sc, voxelize=True, grid=(1, 1, 1))
    for n in (63, 5003, 70001):
        t = tracks(sc, n, n)
        s0, h0 = g.geo_dist_to_boundary(walk, *t, mode=g.GEO_FP64)
        s1, h1 = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)
        assert torch.equal(h0, h1)
        assert torch.equal(s0.view(torch.int64), s1.view(torch.int64))


@pytest.mark.parametrize("mother", ["box", "tube"])
@pytest.mark.parametrize("counts", COUNTS)
def test_point_queries_equal_fp64_bitwise(g, counts, mother):
    """Contains and Safety of points anywhere, on the solids' surfaces and a
    little beside them (where FP32 cannot decide and whole solids are
    evaluated), on their axes and in their coordinate planes."""
    sc = filter_scene(*counts, mother, seed=sum(counts) + 7)
    vol = g.geo_build_volume(sc)
    rng = np.random.default_rng(3)
    for n in (33, 5003, 170001):   # 33 and 5003: 32 points a warp; 170001: 64
        t = tracks(sc, n, n + 1)
        s, _ = g.geo_dist_to_boundary(vol, *t, mode=g.GEO_FP64)
        s = torch.where(torch.isfinite(s), s, 0.0) * (1.0 + 1e-9 * torch.from_numpy(rng.integers(-1, 2, n)).cuda())
        on = [t[k] + s * t[3 + k] for k in range(3)]
        j = rng.integers(0, sc.n_daughters, n)
        axis = sc.trans[j] + np.einsum("nij,nj->ni", sc.rot[j].reshape(n, 3, 3),
                                       rng.uniform(-1.5, 1.5, (n, 3)) * 40.0 * rng.integers(0, 2, (n, 3)))
        axis = [torch.from_numpy(np.ascontiguousarray(axis[:, k])).cuda() for k in range(3)]
        for p in (t[:3], on, axis):
            assert torch.equal(g.geo_contains(vol, *p, mode=g.GEO_FP64), g.geo_contains(vol, *p))
            s0, s1 = g.geo_safety(vol, *p, mode=g.GEO_FP64), g.geo_safety(vol, *p)
            assert torch.equal(s0.view(torch.int64), s1.view(torch.int64))
    assert g.geo_check_device_status(vol) == 0


@pytest.mark.parametrize("n", [33, 4099, 300007])
def test_world_states_equal_fp64_bitwise(g, n):
    """The geometry-tree step from consistent states (Locate, then steps with
    the flags they return) and from arbitrary ones (any node, any flag, any
    point): re-entries and entered nodes that FP32 decides alone give the
    FP64 mode's bits."""
    tree = scenes.world_toy()
    vols = [g.geo_build_volume(s) for s in tree.volumes]
    world = g.geo_build_world(vols, tree.child, tree.root)
    rng = np.random.default_rng(n)
    t = [torch.from_numpy(f).cuda() for f in scenes.world_points(tree, n, n).fields()]
    node = g.geo_world_locate(world, *t[:3])
    flag = torch.full_like(node, -1)

    def both(t, node, flag):
        a = g.geo_world_step(world, *t, node, flag, mode=g.GEO_FP64)
        b = g.geo_world_step(world, *t, node, flag, mode=g.GEO_FP32_REFINE)
        assert torch.equal(a[0].view(torch.int64), b[0].view(torch.int64))
        assert torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])
        return b

    for _ in range(5):
        any_node = torch.from_numpy(rng.integers(-2, world.n_nodes + 2, n).astype(np.int32)).cuda()
        any_flag = torch.from_numpy(rng.integers(-3, 44, n).astype(np.int32)).cuda()
        both(t, any_node, any_flag)
        both(t, node, any_flag)
        s, node2, flag = both(t, node, flag)
        s = torch.where(torch.isfinite(s), s, 0.0)
        t = [t[k] + s * t[3 + k] for k in range(3)] + t[3:]
        if rng.random() < 0.5:   # scattered: another direction from the boundary
            t = t[:3] + [torch.from_numpy(f).cuda() for f in scenes.isotropic(rng, n)]
        node = node2


@pytest.mark.parametrize("n", [1, 33, 4099, 200003, 700001])
@pytest.mark.parametrize("kind,prm", [(scenes.BOX, (3.0, 20.0, 11.0)), (scenes.TUBE, (0.0, 9.0, 14.0)),
                                      (scenes.TUBE, (8.9, 9.0, 4.0)), (scenes.CONE, (5.0, 1.0, 30.0, 20.0, 21.0)),
                                      (scenes.CONE, (30.0, 2.0, 4.0, 9.0, 9.0))])
def test_solid_queries_equal_fp64_bitwise(g, kind, prm, n):
    """One solid's queries against the FP64 kernels of a volume that holds it
    (DistFromOutside) or is it (the others): points near and far beyond the
    reach of its FP32 copies, on its rims and corners and a little beside
    them; 32, 64 and 128 points a warp."""
    rng = np.random.default_rng(n)
    rot, t = scenes.haar_rotation(rng), np.array([7.0, -3.0, 5.0])
    size = max(prm)
    p = rng.uniform(-2.0, 2.0, (n, 3)) * size * np.where(rng.random((n, 1)) < 0.1, 30.0, 1.0)
    m = n // 2
    if kind == scenes.BOX:
        q = np.array(prm) * rng.choice([-1.0, 1.0, 0.4], (m, 3))
    else:
        e, ph = rng.choice([-1.0, 1.0], m), rng.uniform(0.0, 2.0 * np.pi, m)
        ends = (prm[0], prm[1], prm[0], prm[1], prm[2]) if kind == scenes.TUBE else (*prm[1:], prm[0])
        lo, hi = rng.integers(2, size=m), e > 0
        r = np.where(hi, np.where(lo, ends[2], ends[3]), np.where(lo, ends[0], ends[1]))
        q = np.stack([r * np.cos(ph), r * np.sin(ph), e * ends[4]], axis=1)
    p[:m] = q * (1.0 + rng.choice([0.0, 1e-8, 1e-6, 1e-4], (m, 1)) * rng.uniform(-1.0, 1.0, (m, 3)))
    d = np.stack(scenes.isotropic(rng, n), axis=1)
    p -= d * rng.uniform(0.0, 3.0, (n, 1)) * size * rng.integers(0, 2, (n, 1))

    def cuda(a):
        return [torch.from_numpy(np.ascontiguousarray(a[:, k])).cuda() for k in range(3)]

    R = rot.reshape(3, 3)
    placed = cuda(p @ R.T + t) + cuda(d @ R.T)
    hall = g.geo_build_volume(scenes._scene("hall", scenes.BOX, (1e4, 1e4, 1e4), [(kind, prm, rot, t)]))
    step, hit = g.geo_dist_to_boundary(hall, *placed, mode=g.GEO_FP64)
    out, face = g.geo_shape_query(kind, prm, g.GEO_Q_DIST_OUT, *placed, rot=rot, trans=t, want_face=True)
    assert torch.equal(torch.where(hit == 0, step, torch.inf).view(torch.int64), out.view(torch.int64))
    assert torch.equal((face >= 0), (hit == 0) & (step > 0))
    own = cuda(p) + cuda(d)
    solid = g.geo_build_volume(scenes.leaf(kind, prm))
    inside = g.geo_contains(solid, *own[:3], mode=g.GEO_FP64) == -1
    assert torch.equal(g.geo_shape_query(kind, prm, g.GEO_Q_CONTAINS, *own[:3]) == 1.0, inside)
    step, _ = g.geo_dist_to_boundary(solid, *own, mode=g.GEO_FP64)
    out, face = g.geo_shape_query(kind, prm, g.GEO_Q_DIST_IN, *own, want_face=True)
    assert torch.equal(step.view(torch.int64), out.view(torch.int64))
    assert torch.equal(face >= 0, inside)
    saf = g.geo_shape_query(kind, prm, g.GEO_Q_SAFETY_IN, *own[:3])
    assert torch.equal(g.geo_safety(solid, *own[:3], mode=g.GEO_FP64).view(torch.int64), saf.view(torch.int64))
