"""The launch shapes of a sweep (fld_solve_params.temporal_depth, the choice of
the library's autotuner): every one of them updates each unknown with the same
arithmetic, so all give the same state bit for bit.  The reference is the
TMA-blocked kernel with T = 1, whose tiles do not depend on the row length."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid, random_case  # noqa: E402


def state_after(shape, precision, depth, iters, limiter="lp", bf16=0, seed=31):
    sig, alb, j, h = random_case(shape, seed)
    rng = np.random.default_rng(seed)
    padded = tuple(n + 2 for n in shape)
    phi0, D0 = rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)
    with gpu_grid(sig, alb, j, h) as g:
        g.set_state(phi0, D0)
        g.iterate(fld.params(limiter=limiter, precision=precision, omega=1.4, warm_start=1, temporal_depth=depth,
                             medium_bf16=bf16), iters)
        return g.get_state()


# rows of 1, 8, 32, 33, 40 and 64 pairs of one colour: 33 and 40 leave more than
# a sixth of 32-wide tiles idle and run by item number, 32 and 64 do not
@pytest.mark.parametrize("nx", [1, 31, 128, 129, 131, 160, 256])
@pytest.mark.parametrize("precision,bf16", [("fp32", 0), ("pair", 1)])
def test_launched_passes_by_row_length(nx, precision, bf16):
    shape = (5, 7, nx)
    want = state_after(shape, precision, 1, 4, bf16=bf16)
    got = state_after(shape, precision, -1, 4, bf16=bf16)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


# Forms that the tuner picks on small grids, chosen here through a tuning cache
# that names them: whole iterations per launch (-4), one unknown per thread (-5;
# -2 in the float-float family, which has no -4).  Single rows and planes, rows whose first or last unknown is of
# either colour, tiles cut at the far faces, an odd iteration left to the passes
ROWS_SHAPES = [(1, 1, 1), (1, 1, 9), (9, 1, 6), (1, 40, 3), (2, 3, 2), (7, 9, 8), (17, 33, 31), (24, 24, 24),
               (32, 32, 32), (40, 37, 33), (5, 6, 250)]
FAMILIES = {"fp32": 0, "pair": 3, "mixed": 1}
_CHILD = """
import sys, numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import test_gpu_sweep_shapes as t
out = {{}}
for shape in t.ROWS_SHAPES:
    for precision in t.FAMILIES:
        for limiter, bf16 in (("lp", 0), ("larsen", 1)):
            if precision == "mixed" and bf16:
                bf16 = 0
            for depth in (0, -1):
                phi, D = t.state_after(shape, precision, depth, 5, limiter, bf16)
                out["%s %s %s %d phi" % (shape, precision, limiter, depth)] = phi
                out["%s %s %s %d D" % (shape, precision, limiter, depth)] = D
np.savez({path!r}, **out)
"""


@pytest.mark.parametrize("form", [-4, -5])
def test_small_grid_forms_equal_the_pair_passes(tmp_path, form):
    import os
    import subprocess
    import sys

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lines = ["v6 %dx%dx%d fam%d lim%d r2 bf%d sm%d | %d 1 64 0 0 0"
             % (s[2], s[1], s[0], fam, lim, bf, sms, -2 if fam == 1 else form)
             for s in ROWS_SHAPES for fam in (0, 1, 3) for lim in (fld.LIMITERS["lp"], fld.LIMITERS["larsen"])
             for bf in (0, 1)]
    cache = tmp_path / "tune.txt"
    cache.write_text("\n".join(lines) + "\n")
    path = str(tmp_path / "states.npz")
    tests = os.path.dirname(os.path.abspath(__file__))
    code = _CHILD.format(root=os.path.dirname(tests), tests=tests, path=path)
    subprocess.run([sys.executable, "-c", code], check=True, timeout=600,
                   env=dict(os.environ, FLD_TUNE_CACHE=str(cache)))
    assert len(cache.read_text().splitlines()) == len(lines)      # nothing was tuned: every form above was the one run
    got = np.load(path)
    for key in got.files:
        if " 0 " in key:
            assert np.array_equal(got[key], got[key.replace(" 0 ", " -1 ")]), key


# Every family the tuner times, on the legacy default stream (handle 1), which
# cannot be captured: shapes that nothing else here has tuned
@pytest.mark.parametrize("precision,shape", [("fp32", (6, 13, 19)), ("pair", (6, 13, 21)), ("mixed", (6, 13, 23))])
def test_tuning_on_the_legacy_stream(precision, shape):
    sig, alb, j, h = random_case(shape, 31)
    want = state_after(shape, precision, -1, 5)
    rng = np.random.default_rng(31)
    padded = tuple(n + 2 for n in shape)
    phi0, D0 = rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)
    nz, ny, nx = shape
    with fld.Grid(nx, ny, nz, h, stream=1) as g:
        g.set_medium(sig, alb)
        g.set_source(j)
        g.set_state(phi0, D0)
        g.iterate(fld.params(limiter="lp", precision=precision, omega=1.4, warm_start=1), 5)
        got = g.get_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])


# Ticks: the third and later calls of fld_iterate with one count and set of
# parameters replay a graph on a small grid; a changed count or parameter, a
# state set between the calls, a caller's own capture and the legacy stream
# leave the bits of plain launches (temporal_depth -1 on a grid of its own each)
@pytest.mark.parametrize("precision,bf16", [("fp32", 0), ("pair", 1), ("mixed", 0)])
@pytest.mark.parametrize("legacy", [0, 1])
def test_repeated_iterate_replays_the_same_bits(precision, bf16, legacy):
    shape = (11, 14, 37)
    sig, alb, j, h = random_case(shape, 7)
    rng = np.random.default_rng(7)
    padded = tuple(n + 2 for n in shape)
    states = [(rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)) for _ in range(2)]
    nz, ny, nx = shape

    def par(omega, depth):
        return fld.params(precision=precision, omega=omega, warm_start=1, temporal_depth=depth, medium_bf16=bf16)

    stream = torch.cuda.Stream()
    with fld.Grid(nx, ny, nz, h, stream=1 if legacy else stream.cuda_stream) as g, gpu_grid(sig, alb, j, h) as ref:
        g.set_medium(sig, alb)
        g.set_source(j)
        calls = [(5, 1.4)] * 5 + [(6, 1.4)] * 4 + [(6, 1.2)] * 4 + [(5, 1.4)] * 3
        for s, (phi0, D0) in enumerate(states):
            g.set_state(phi0, D0)
            ref.set_state(phi0, D0)
            for n, omega in calls:
                g.iterate(par(omega, 0), n)
                ref.iterate(par(omega, -1), n)
        if not legacy:
            torch.cuda.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                g.iterate(par(1.4, 0), 5)
            graph.replay()
            torch.cuda.synchronize()
            ref.iterate(par(1.4, -1), 5)
        got, want = g.get_state(), ref.get_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
