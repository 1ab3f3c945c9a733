"""The light march along thin rows between dense ones: at a voxel centre the
blend of two corners is the corner itself, whichever side of the other it lies
on, so a thin row's optical depth holds none of its neighbours' rounding.
Reference: the oracle (FP64), voxel by voxel."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid  # noqa: E402

# an optical depth of 0.3 from samples each within three roundings (2e-7), the
# transmittance and three products: 1e-6 with a factor of two in hand
TOL = 1e-6


# rays along each axis, both ways; thin rows of even and of odd index, the
# outermost ones among them; an axis of one voxel (the general corner search)
@pytest.mark.parametrize("thin", [0, 1])
@pytest.mark.parametrize("axis,sign", [(0, 1), (0, -1), (1, 1), (1, -1), (2, 1)])
@pytest.mark.parametrize("flat", [0, 1])
def test_thin_rows_between_dense_ones(axis, sign, thin, flat):
    n = [24, 24, 24]                                   # z, y, x
    ray = 2 - axis
    other = [a for a in range(3) if a != ray]
    n[other[0]], n[other[1]] = (1 if flat else 6), 8
    idx = np.indices(n)
    row = idx[other[1]] if flat else idx[other[0]] + idx[other[1]]
    sig = np.where(row % 2 == thin, 1e-3, 1e4).astype(np.float32)
    alb = np.full(n, 0.5, np.float32)
    h = 10.0
    direction = [0.0, 0.0, 0.0]
    direction[axis] = float(sign)
    want = oracle.bake_directional(sig, alb, h, direction, 1.5)
    with gpu_grid(sig, alb, np.zeros(n, np.float32), h) as g:
        g.bake_directional(direction, 1.5)
        got = g.get_source()
    rows = sig < 1.0
    assert (np.abs(got - want)[rows] <= TOL * want[rows]).all()
