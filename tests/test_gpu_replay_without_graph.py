"""fld_iterate where no graph can be made (its instantiation fails for want of
memory): the call goes on with launches, with the same bits, whether the graph
is that of a replay or those a new shape's forms are timed by.  The failure is
a fake of cudaGraphInstantiate, preloaded into a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

# cudaGraphInstantiate with error 2 (cudaErrorMemoryAllocation) while told so
_FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
static int refuse = 0, refusals = 0;
void fake_refuse(int on) { refuse = on; }
int fake_refusals(void) { return refusals; }
int cudaGraphInstantiate(void **exec, void *graph, unsigned long long flags) {
    static int (*next)(void **, void *, unsigned long long) = 0;
    if (refuse) { ++refusals; return 2; }
    if (!next) next = (int (*)(void **, void *, unsigned long long))dlsym(RTLD_NEXT, "cudaGraphInstantiate");
    return next(exec, graph, flags);
}
"""

_CHILD = """
import ctypes, sys, numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import test_gpu_replay as t
fake = ctypes.CDLL({fake!r})
# a shape that was never tuned, and cannot be: no candidate's graph can be made
import os
os.environ["FLD_TUNE_CACHE"] = {cache!r}
fake.fake_refuse(1)
first = []
with t.grid(None) as g:
    g.iterate(t.par(1.4, "pair"), 8)
    first.append(g.get_state())
fake.fake_refuse(0)
assert not os.path.exists({cache!r})
with t.grid(None) as g:
    g.iterate(t.par(1.4, "pair"), 8)          # tuned now
    first.append(g.get_state())
assert os.path.exists({cache!r})
assert np.array_equal(first[0][0], first[1][0]) and np.array_equal(first[0][1], first[1][1])
start = fake.fake_refusals()
with t.grid(None) as g, t.grid(None) as ref:
    for x in (g, ref):
        for n in (8, 3, 2):
            x.iterate(t.par(1.4), n)          # every form tuned
    fake.fake_refuse(1)
    for k in range(6):
        g.iterate(t.par(1.4), 8)
        for n in (3, 3, 2):
            ref.iterate(t.par(1.4), n)
        a, b = g.get_state(), ref.get_state()
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]), k
    assert fake.fake_refusals() == start + 1          # asked for once, not on every call
    fake.fake_refuse(0)
    for k in range(4):                        # another count: graphs again
        g.iterate(t.par(1.4), 5)
        for n in (3, 2):
            ref.iterate(t.par(1.4), n)
    a, b = g.get_state(), ref.get_state()
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
print("done")
"""


def test_launches_go_on_where_no_graph_can_be_made(tmp_path):
    src, so = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(_FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    tests = os.path.dirname(os.path.abspath(__file__))
    code = _CHILD.format(root=os.path.dirname(tests), tests=tests, fake=str(so), cache=str(tmp_path / "tune.txt"))
    r = subprocess.run([sys.executable, "-c", code], timeout=600, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=str(so)))
    assert r.returncode == 0, r.stderr[-2000:]
    assert "done" in r.stdout
