"""The forms the tuner picks for small grids, run as a solve runs them: from graphs
of a whole block, launched early or not.  Each is named in a tuning cache and
compared with the pair passes (temporal_depth -1), bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid, random_case  # noqa: E402

# the smallest, single rows, odd edges, rows cut at the far faces, more CTAs than are
# settled (1216 of 128 unknowns)
SHAPES = [(1, 1, 1), (1, 1, 9), (2, 3, 2), (17, 33, 31), (32, 32, 32), (5, 6, 250), (70, 72, 76)]
FAMILIES = {"fp32": 0, "pair": 3, "mixed": 1}
CASES = [("lp", 0), ("kershaw", 0), ("larsen", 1), ("sum", 0)]
BLOCK = 20            # iterations of a graph: 40 passes, five that settle


def state_after(shape, precision, limiter, bf16, depth):
    """A state after two blocks: of a solve; float-float passes, which a solve
    reaches only after others, in the replays of equal fld_iterate calls (the
    pair passes: in calls too short to be replayed)."""
    sig, alb, j, h = random_case(shape, 5)
    rng = np.random.default_rng(5)
    padded = tuple(n + 2 for n in shape)
    p = fld.params(limiter=limiter, precision=precision, omega=1.4, warm_start=1, temporal_depth=depth,
                   medium_bf16=bf16, tol=0.0, max_iters=2 * BLOCK, check_every=BLOCK)
    with gpu_grid(sig, alb, j, h) as g:
        g.set_state(rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded))
        if precision != "mixed":
            g.solve(p, check=False)
        else:
            for count in [BLOCK] * 4 if depth == 0 else [2] * (2 * BLOCK):
                g.iterate(p, count)
        return g.get_state()


_CHILD = """
import sys, numpy as np
sys.path[:0] = [{root!r}, {tests!r}]
import test_gpu_solve_forms as t
for shape in t.SHAPES:
    for precision in t.FAMILIES:
        for limiter, bf16 in t.CASES:
            if precision == "mixed" and bf16:
                bf16 = 0
            got, want = (t.state_after(shape, precision, limiter, bf16, depth) for depth in (0, -1))
            assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), (shape, precision, limiter)
print("done")
"""


# pairs in tiles, by running number, quads, whole iterations, one unknown (float-float:
# two unknowns with seven and with five CTAs per SM, one), early and not
@pytest.mark.parametrize("form", [-1, -3, -2, -4, -5])
@pytest.mark.parametrize("early", [1, 0])
def test_form_in_a_graph_equals_the_pair_passes(tmp_path, form, early):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    lines = ["v6 %dx%dx%d fam%d lim%d r2 bf%d sm%d | %d %d 64 1 1 1"
             % (s[2], s[1], s[0], fam, fld.LIMITERS[lim], bf, sms, form if fam != 1 else max(form, -3), early)
             for s in SHAPES for fam in FAMILIES.values() for lim in ("lp", "kershaw", "larsen", "sum")
             for bf in (0, 1)]
    cache = tmp_path / "tune.txt"
    cache.write_text("\n".join(lines) + "\n")
    tests = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, "-c", _CHILD.format(root=os.path.dirname(tests), tests=tests)],
                       capture_output=True, text=True, timeout=900, env=dict(os.environ, FLD_TUNE_CACHE=str(cache)))
    assert r.returncode == 0, r.stderr[-2000:]
    assert "done" in r.stdout
    assert len(cache.read_text().splitlines()) == len(lines)      # nothing was tuned: the named form ran
