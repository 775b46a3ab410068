"""A one-solid query allocates nothing on the host: with every operator new of
the library failing, the queries still run (a C entry must not end in an
exception)."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HOOK = r"""
#include <dlfcn.h>
#include <cstdlib>
#include <cstring>
#include <new>
static thread_local int armed = 0;
extern "C" void hook_arm(int on) { armed = on; }
void* operator new(std::size_t n) {
    if (armed) {
        Dl_info i;
        if (dladdr(__builtin_return_address(0), &i) && i.dli_fname && std::strstr(i.dli_fname, "libgeonav"))
            throw std::bad_alloc();
    }
    if (void* p = std::malloc(n ? n : 1)) return p;
    throw std::bad_alloc();
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""

RUN = r"""
import ctypes, sys
import torch
import paper_1312_0816_gb300 as g
from paper_1312_0816_gb300 import scenes
hook = ctypes.CDLL(sys.argv[1])
g.load()
pc = scenes.Pcon((-30.0, -20.0, 20.0, 30.0), (0.0, 5.0, 5.0, 0.0), (25.0, 10.0, 10.0, 25.0))
solids = ((scenes.BOX, (30.0, 20.0, 40.0)), (scenes.TUBE, (10.0, 40.0, 50.0)), (scenes.CONE, (40.0, 10.0, 30.0, 20.0, 45.0)),
          (scenes.PCON, pc))
for n in (100, 100000):
    t = [torch.rand(n, dtype=torch.float64, device="cuda") * 100.0 - 50.0 for _ in range(6)]
    for kind, prm in solids:
        for what in (g.GEO_Q_DIST_OUT, g.GEO_Q_DIST_IN, g.GEO_Q_SAFETY_OUT, g.GEO_Q_SAFETY_IN, g.GEO_Q_CONTAINS):
            q = t if what in (g.GEO_Q_DIST_OUT, g.GEO_Q_DIST_IN) else t[:3]
            a = g.geo_shape_query(kind, prm, what, *q)
            hook.hook_arm(1)
            b = g.geo_shape_query(kind, prm, what, *q)
            hook.hook_arm(0)
            assert torch.equal(a.view(torch.int64), b.view(torch.int64))
print("ran")
"""


def test_queries_allocate_nothing(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, so = tmp_path / "hook.cpp", tmp_path / "hook.so"
    src.write_text(HOOK)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-o", str(so), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", RUN, str(so)], cwd=ROOT, env={**os.environ, "LD_PRELOAD": str(so)},
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "ran" in r.stdout, r.stderr[-2000:]
