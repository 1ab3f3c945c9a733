"""FP64 sweeps over media whose extinction floor is far below any physical one:
D = F / sigma' reaches 1e150 and more in vacuum, and no product of the update
leaves the range of a double.  Reference: the oracle (FP64), one iteration."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid, oracle_problem, random_case, rel_el  # noqa: E402


# extinction floors around 1e-154, below which D squared overflows; local rounds 2 (the
# fast path) and 3
@pytest.mark.parametrize("limiter", ["lp", "kershaw", "larsen", "cda"])
@pytest.mark.parametrize("floor", [1e-3, 1e-150, 1e-160, 1e-200])
@pytest.mark.parametrize("local", [2, 3])
def test_one_iteration_with_a_tiny_extinction_floor(limiter, floor, local):
    sig, alb, j, h = random_case((7, 9, 8), 12)
    rng = np.random.default_rng(12)
    padded = tuple(n + 2 for n in sig.shape)
    phi0, D0 = rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)
    ref = oracle_problem(sig, alb, j, h, limiter=limiter, omega=1.4, local_iters=local, nthreads=1, sigma_eps=floor)
    oracle.init_state(ref)
    ref.phi[...], ref.D[...] = phi0, D0
    oracle.rb_iteration(ref, 1)
    assert np.isfinite(ref.phi).all() and np.isfinite(ref.D).all()
    with gpu_grid(sig, alb, j, h) as g:
        g.set_state(phi0, D0)
        g.iterate(fld.params(limiter=limiter, precision="fp64", omega=1.4, local_iters=local, warm_start=1,
                             sigma_eps=floor), 1)
        phi, D = g.get_state()
    # D spans 150 orders: each element against its own size
    assert rel_el(phi, ref.phi, also=phi0) <= 1e-12
    assert (np.abs(D - ref.D) <= 1e-11 * np.abs(ref.D)).all()
