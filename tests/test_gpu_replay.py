"""fld_iterate on small grids replays a graph from the third equal call on: the
bits are those of passes launched one by one, call by call, and the call only
enqueues, whatever changed since the last one."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import random_case  # noqa: E402

SHAPE = (11, 14, 37)


def grid(stream):
    sig, alb, j, h = random_case(SHAPE, 7)
    nz, ny, nx = SHAPE
    g = fld.Grid(nx, ny, nz, h, stream=stream)
    g.set_medium(sig, alb)
    g.set_source(j)
    rng = np.random.default_rng(7)
    padded = tuple(n + 2 for n in SHAPE)
    g.set_state(rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded))
    return g


def par(omega, precision="fp32", depth=0, **kw):
    return fld.params(precision=precision, omega=omega, warm_start=1, temporal_depth=depth, **kw)


# half a second of work ahead on the stream: a call that waits for it takes as long
def test_a_changed_parameter_does_not_wait_for_the_stream():
    stream = torch.cuda.Stream()
    with grid(stream.cuda_stream) as g, grid(torch.cuda.Stream().cuda_stream) as ref:
        for omega, n in ((1.4, 8), (1.3, 8), (1.3, 6)):      # every form tuned
            g.iterate(par(omega), n)
            ref.iterate(par(omega), n)
        for _ in range(4):
            g.iterate(par(1.4), 8)
            ref.iterate(par(1.4, depth=-1), 3)
            ref.iterate(par(1.4, depth=-1), 3)
            ref.iterate(par(1.4, depth=-1), 2)
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(1_000_000_000)
        t = time.perf_counter()
        g.iterate(par(1.4), 8)                               # a replay that is still waiting
        g.iterate(par(1.2), 8)
        g.iterate(par(1.2), 6)
        took = time.perf_counter() - t
        assert not stream.query()
        assert took < 0.2
        for omega, n in ((1.4, 8), (1.2, 8), (1.2, 6)):
            for k in (3, 3, n - 6):
                ref.iterate(par(omega, depth=-1), k)
        got, want = g.get_state(), ref.get_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
