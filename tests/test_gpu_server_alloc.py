"""A server whose device memory runs out as a grid joins: the addition reports
it, and the steps of the grids that run go on to the bits of their solo solves.
The failing allocation is a fake of cudaMalloc, preloaded into a process of its
own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

# cudaMalloc with error 2 (cudaErrorMemoryAllocation) for two sizes
_FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static size_t refused[2] = {0, 0};
void fake_refuse(size_t a, size_t b) { refused[0] = a; refused[1] = b; }
int cudaMalloc(void **p, size_t n) {
    static int (*next)(void **, size_t) = 0;
    if (n && (n == refused[0] || n == refused[1])) return 2;
    if (!next) next = (int (*)(void **, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
    return next(p, n);
}
"""

_CHILD = """
import ctypes, sys, numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import paper_1403_8105_gb300 as fld
import test_gpu_server as t
fake = ctypes.CDLL({fake!r})
fake.fake_refuse.argtypes = [ctypes.c_size_t] * 2
p = fld.params(limiter="lp", precision="mixed", tol=1e-6, check_every=32, max_iters=200000, anderson=4)
shapes = [(12, 12, 12), (9, 10, 11), (8, 14, 10), (10, 10, 10), (11, 9, 12), (9, 9, 9)]
grids = [t._grid(a, s) for a, s in enumerate(shapes)]
want = []
for a, s in enumerate(shapes):
    with t._grid(a, s) as g:
        g.solve(p)
        want.append(g.get_state()[0])
with fld.Server(p) as srv:
    for a in range(5):
        srv.add(grids[a], a)
    # room for the dot products (16 doubles a grid) of 5 + 2 + 4 and of 6 + 3 + 4 grids
    fake.fake_refuse(8 * 16 * 11, 8 * 16 * 13)
    done = set(tag for tag, _ in srv.step())
    left = set(range(5))
    try:
        srv.add(grids[5], 5)
        left.add(5)
    except fld.FldError:
        print("refused")
    while srv.active:
        done |= set(tag for tag, _ in srv.step())
    assert done == left, done
    fake.fake_refuse(0, 0)
    if 5 not in left:
        srv.add(grids[5], 5)
        while srv.active:
            srv.step()
for g, w in zip(grids, want):
    assert np.array_equal(g.get_state()[0], w)
    g.close()
"""


def test_memory_runs_out_as_a_grid_joins(tmp_path):
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(_FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    tests = os.path.dirname(os.path.abspath(__file__))
    code = _CHILD.format(root=os.path.dirname(tests), tests=tests, fake=str(so))
    r = subprocess.run([sys.executable, "-c", code], timeout=600, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr[-2000:]
    assert "refused" in r.stdout
