"""A batch whose waits for staged tables run out: the tracks take the FP64
routines instead of reading tables that may not be there, and the status words
say so."""
import numpy as np
import pytest

from paper_1312_0816_gb300 import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ST_TMA_TIMEOUT = 1


@pytest.fixture(scope="module")
def g():
    import paper_1312_0816_gb300 as pkg

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.load()
    return pkg


def boxes_and_a_segment(n, rng):
    rows = [(scenes.BOX, rng.uniform(2.0, 6.0, 3), scenes.haar_rotation(rng), rng.uniform(-90.0, 90.0, 3)) for _ in range(n)]
    rows.append((scenes.TUBS, (2.0, 9.0, 9.0, 0.3, 4.0), np.eye(3).reshape(9), (0.0, 0.0, 0.0)))
    return scenes._scene(f"seg{n}", scenes.BOX, (100.0,) * 3, rows)


@pytest.mark.parametrize("tile", [384, 256])
@pytest.mark.parametrize("daughters", [3, 250])   # two volumes' tables side by side, and one at a time
def test_batch_without_its_tables(g, daughters, tile):
    rng = np.random.default_rng(daughters)
    vols = [g.geo_build_volume(boxes_and_a_segment(n, rng)) for n in (daughters, daughters - 1, 2)]
    n = 400011
    p = rng.uniform(-101.0, 101.0, (3, n))   # some outside
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (*p, *np.stack(scenes.isotropic(rng, n)))]
    t[3][7] = float("nan")
    cuts = [0, 17, 400, n // 3, n // 2, n - 5000, n]
    batch = g.geo_build_batch(vols, [(k % 3, a, b - a) for k, (a, b) in enumerate(zip(cuts, cuts[1:]))], tile_tracks=tile)
    ref = g.geo_dist_to_boundary_batched(batch, *t)
    assert all(g.geo_check_device_status(v) == 0 for v in vols)
    out = g.geo_selftest_batch_timeout(batch, *t)
    assert torch.equal(out[0].view(torch.int64), ref[0].view(torch.int64)) and torch.equal(out[1], ref[1])
    for v in vols:
        with pytest.raises(g.GeoError) as e:
            g.geo_check_device_status(v)
        assert e.value.status == 5 and "0x1" in str(e.value)
    again = g.geo_dist_to_boundary_batched(batch, *t)
    assert torch.equal(again[0].view(torch.int64), ref[0].view(torch.int64)) and torch.equal(again[1], ref[1])
    assert all(g.geo_check_device_status(v) == 0 for v in vols)
