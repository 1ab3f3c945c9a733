"""Point lights so far away that the square of their distance, in voxels or in
the world's unit, leaves the range of a float: the march still finds its
direction and its end.  Reference: the oracle (FP64)."""
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


# voxel edge, distance of the light: near; its square beyond a float in voxels
# only; in the world's unit too; the position itself beyond a float in voxels
@pytest.mark.parametrize("h,dist", [(1.0 / 33, 1e3), (1e-3, 1e17), (1.0 / 33, 1e19), (1e3, 1e21), (1e-20, 1e12),
                                    (1e-25, 1e17)])
@pytest.mark.parametrize("direction", [(0.2, -0.7, 0.68), (0.0, 0.0, 1.0), (-1.0, 1e-3, 0.0)])
def test_far_point_light(h, dist, direction):
    shape = (17, 20, 33)
    sig, alb, j, h0 = random_case(shape, 9)
    sig = (sig.astype(np.float64) * (h0 / h)).astype(np.float32)      # the same optical depths
    d = np.array(direction) / np.linalg.norm(direction)
    pos = tuple(float(x) for x in dist * d)
    power = min(1e38, 4.0 * np.pi * dist * dist) / max(1.0, float(sig.max()))     # times sigma_s within a float
    want = oracle.bake_point(sig, alb, h, pos, power)
    with gpu_grid(sig, alb, j, h) as g:
        g.bake_point(pos, power)
        got = g.get_source()
    assert np.abs(got - want).max() <= TOL * np.abs(want).max()
