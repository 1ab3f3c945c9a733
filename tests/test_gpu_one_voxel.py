"""Grids of one voxel, whose black pass has no unknown: passes that follow one
another early keep their order, so a run of iterations equals single ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid  # noqa: E402


def one(shape, sigma=3.0):
    full = [np.full(shape, v, np.float32) for v in (sigma, 0.8, 1.7)]
    return gpu_grid(*full, 0.25)


def start(shape):
    rng = np.random.default_rng(4)
    padded = tuple(n + 2 for n in shape)
    return rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)


# one voxel, and the smallest grids with unknowns of both colours
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 1, 2), (2, 1, 1)])
@pytest.mark.parametrize("precision", ["fp64", "fp32", "pair", "mixed"])
@pytest.mark.parametrize("depth", [0, -1])
def test_iterations_in_a_row_equal_single_ones(shape, precision, depth):
    p = fld.params(precision=precision, omega=1.3, warm_start=1, temporal_depth=depth)
    got = []
    for calls, count in ((1, 48), (48, 1)):
        with one(shape) as g:
            g.set_state(*start(shape))
            for _ in range(calls):
                g.iterate(p, count)
            got.append(g.get_state())
    assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])


@pytest.mark.parametrize("precision", ["fp32", "pair"])
@pytest.mark.parametrize("batch_launch", [0, 1])
def test_batch_of_one_voxel_grids(precision, batch_launch):
    p = fld.params(precision=precision, omega=1.3, tol=0.0, max_iters=96, check_every=32, batch_launch=batch_launch)
    solo = []
    for sigma in (1.0, 3.0, 9.0):
        with one((1, 1, 1), sigma) as g:
            g.solve(p, check=False)
            solo.append(g.get_state()[0])
    grids = [one((1, 1, 1), sigma) for sigma in (1.0, 3.0, 9.0)]
    try:
        fld.fld_solve_batch(grids, p, check=False)
        for g, want in zip(grids, solo):
            assert np.array_equal(g.get_state()[0], want)
    finally:
        for g in grids:
            g.close()
