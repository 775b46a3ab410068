"""Two host threads that call the same kernel on volumes of different table
sizes, each on its own stream."""
import threading

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


@pytest.mark.parametrize("query", ["contains", "safety", "step"])
def test_two_table_sizes(g, query):
    rng = np.random.default_rng(1)

    def boxes(n):
        return scenes._scene(f"boxes{n}", scenes.BOX, (400.0,) * 3,
                             [(scenes.BOX, rng.uniform(1.0, 5.0, 3), np.eye(3).reshape(9), rng.uniform(-390.0, 390.0, 3))
                              for _ in range(n)])

    # staged tables of 33 to 36 KB for the step, 40 and 86 KB for the points' queries
    vols = [g.geo_build_volume(boxes(n)) for n in ((229, 250) if query == "step" else (277, 600))]
    n = 40000 if query == "step" else 33000
    t = [torch.from_numpy(a).cuda() for a in (*rng.uniform(-390.0, 390.0, (3, n)), *np.stack(scenes.isotropic(rng, n)))]

    def call(v, out, stream=None):
        if query == "contains":
            return g.geo_contains(v, *t[:3], where=out[1], stream=stream)
        if query == "safety":
            return g.geo_safety(v, *t[:3], safety=out[0], stream=stream)
        return g.geo_dist_to_boundary(v, *t, step=out[0], hit=out[1], stream=stream)

    outs = [(torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")) for _ in range(2)]
    for v, o in zip(vols, outs):
        call(v, o)
    ref = [(o[0].clone(), o[1].clone()) for o in outs]
    torch.cuda.synchronize()
    failed, start = [], threading.Barrier(2)

    def go(k):
        s = torch.cuda.Stream()
        start.wait()
        for _ in range(4000):
            try:
                call(vols[k], outs[k], stream=s)
            except g.GeoError as e:
                failed.append(str(e))
                return
        s.synchronize()

    th = [threading.Thread(target=go, args=(k,)) for k in range(2)]
    for x in th:
        x.start()
    for x in th:
        x.join()
    torch.cuda.synchronize()
    assert not failed
    for o, r in zip(outs, ref):
        assert torch.equal(o[0].view(torch.int64), r[0].view(torch.int64)) and torch.equal(o[1], r[1])
