"""Tracks whose first two tasks are all but tied: thin slabs on the mother's
walls, of such a thickness that the bound of the entry into a slab and that of
the mother's exit are equal up to their rounding.  They are the tracks that
the grid's and the batch's kernels take through the FP32 pass a second time."""
import math

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


@pytest.mark.parametrize("seed", [0, 1])
def test_tied_bounds(g, seed):
    rng = np.random.default_rng(seed)
    half, eps = 100.0, 2.0 ** -24
    rows = []
    for _ in range(300):
        k = rng.integers(3)
        size = np.full(3, rng.uniform(5.0, 30.0))
        size[k] = 8.0 * eps * (half * math.sqrt(3.0) - 30.0) * rng.uniform(0.2, 2.0)   # the inflations' difference
        at = rng.uniform(-70.0, 70.0, 3)
        at[k] = rng.choice([-1.0, 1.0]) * (half - size[k] - 1e-7 * rng.integers(0, 3))
        rows.append((scenes.BOX, size, np.eye(3).reshape(9), at))
    sc = scenes._scene("slabs", scenes.BOX, (half,) * 3, rows)
    flat = g.geo_build_volume(sc)
    n = 1 << 20
    p = rng.uniform(-0.99 * half, 0.99 * half, (3, n))
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p, *np.stack(scenes.isotropic(rng, n)))]
    s, h = g.geo_dist_to_boundary(flat, *t, mode=g.GEO_FP64)

    def check(out):
        assert torch.equal(s.view(torch.int64), out[0].view(torch.int64)) and torch.equal(h, out[1])

    check(g.geo_dist_to_boundary(flat, *t))
    grids = [g.geo_build_volume(sc, voxelize=True, grid=c) for c in ((4, 4, 4), (48, 48, 48))]   # staged, in global memory
    for v in grids:
        check(g.geo_dist_to_boundary(v, *t))
    check(g.geo_dist_to_boundary_batched(g.geo_build_batch([flat], [(0, 0, n)]), *t))
    check(g.geo_dist_to_boundary_batched(g.geo_build_batch([grids[0], flat], [(0, 0, n // 2), (1, n // 2, n - n // 2)]), *t))
