"""The light march at the sizes where its corner search can go wrong: axes of
one and two voxels, rays that leave through every face, lights inside the grid
and at a voxel centre, steps longer than the grid.  Reference: the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid, random_case  # noqa: E402

# single-precision coordinates: an optical depth of up to ~30 from ~100 samples,
# each to a few 1e-7 of the medium's largest value
TOL = 2e-5


@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 9, 4), (6, 1, 1), (2, 2, 2), (17, 20, 33)])
@pytest.mark.parametrize("direction", [(1, 0, 0), (0, 0, 1), (0.3, -0.8, -0.5), (-0.3, 0.8, 0.5)])
def test_directional(shape, direction):
    sig, alb, j, h = random_case(shape, 3)
    want = oracle.bake_directional(sig, alb, h, direction, 1.5)
    with gpu_grid(sig, alb, j, h) as g:
        g.bake_directional(direction, 1.5)
        got = g.get_source()
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()
    assert not got[sig == 0].any()


@pytest.mark.parametrize("shape", [(1, 9, 4), (2, 2, 2), (17, 20, 33)])
@pytest.mark.parametrize("where", [(0.5, 0.4, 1.3), (0.31, 0.4, 0.6), "centre"])
def test_point(shape, where):
    sig, alb, j, h = random_case(shape, 4)
    nz, ny, nx = shape
    pos = ((nx // 2 + 0.5) * h, (ny // 2 + 0.5) * h, (nz // 2 + 0.5) * h) if where == "centre" else \
        (where[0] * nx * h, where[1] * ny * h, where[2] * nz * h)
    want = oracle.bake_point(sig, alb, h, pos, 3.0)
    with gpu_grid(sig, alb, j, h) as g:
        g.bake_point(pos, 3.0)
        got = g.get_source()
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()


# steps so short that the count of samples is kept in whole numbers (2^20 of them
# span less than twice the longest axis), against steps a little longer, which
# count in float: the two depths differ by rounding only
def test_sample_count_forms():
    sig, alb, j, h = random_case((2, 3, 2), 5)
    got = []
    for step in (5.6e-6, 5.8e-6):
        with gpu_grid(sig, alb, j, h) as g:
            g.bake_directional((0.2, 0.9, 0.1), 1.5, step * h)
            got.append(g.get_source())
    assert np.abs(got[0] - got[1]).max() <= TOL * np.abs(got[1]).max()
