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
