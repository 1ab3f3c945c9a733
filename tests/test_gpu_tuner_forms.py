"""What the first call on a new shape times: each form once, launches that are
not early only for the fastest launched pass of a small grid, and the
float-float family only where more than one of its forms can be the fastest.
Counted by a cudaGraphInstantiate of the test's own, preloaded into a process."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

_COUNT = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static int made = 0;
int graphs_made(void) { return made; }
int cudaGraphInstantiate(void **exec, void *graph, unsigned long long flags) {
    static int (*next)(void **, void *, unsigned long long) = 0;
    if (!next) next = (int (*)(void **, void *, unsigned long long))dlsym(RTLD_NEXT, "cudaGraphInstantiate");
    ++made;
    return next(exec, graph, flags);
}
"""

_CHILD = """
import ctypes, sys
sys.path[:0] = [{root!r}, {tests!r}]
import paper_1403_8105_gb300 as fld
from test_gpu_parity import gpu_grid, random_case
count = ctypes.CDLL({so!r}).graphs_made
def first_call(shape, precision, limiter):
    before = count()
    with gpu_grid(*random_case(shape, 3)) as g:
        g.iterate(fld.params(precision=precision, limiter=limiter), 1)
    return count() - before
small, large = (12, 14, 16), (80, 88, 96)
a, b = first_call(large, "fp32", "lp"), first_call(small, "fp32", "lp")
# three launched passes and the blocked forms; and one unknown, whole iterations, one not early
assert b == a + 3, (a, b)
assert first_call(small, "mixed", "kershaw") == 2 * b + 3       # two float-float forms, one of them not early
assert first_call(large, "mixed", "kershaw") == 2 * a
lines = open({cache!r}).read().splitlines()
assert len(lines) == 7 and not [l for l in lines if " fam1 " in l and "96x88x80" in l], lines
print("done")
"""


def test_forms_timed_by_a_first_call(tmp_path):
    src, so = tmp_path / "count.c", tmp_path / "count.so"
    src.write_text(_COUNT)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    tests = os.path.dirname(os.path.abspath(__file__))
    cache = str(tmp_path / "tune.txt")
    code = _CHILD.format(root=os.path.dirname(tests), tests=tests, so=str(so), cache=cache)
    r = subprocess.run([sys.executable, "-c", code], timeout=600, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(so), FLD_TUNE_CACHE=cache))
    assert r.returncode == 0, r.stderr[-2000:]
    assert "done" in r.stdout
