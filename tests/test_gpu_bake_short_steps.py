"""The light march in steps so short that a ray takes a hundred thousand samples:
the sum of equal samples stays as accurate as one of them.  Reference: the
exponential of a homogeneous medium's optical depth (FP64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import gpu_grid  # noqa: E402

# the exponential to two units in the last place and three products, 5e-7, and the
# depth itself (up to 29) to a few 1e-9: 1.5e-6 with room
TOL = 1.5e-6


# steps of a power of two of the voxel, so that depth and step are exact; four
# samples are summed at a time: counts of every remainder; both corner searches
@pytest.mark.parametrize("sigma", [13.7, 29.1])
@pytest.mark.parametrize("per_voxel", [2, 6, 1024, 2048])
@pytest.mark.parametrize("nz", [1, 2])
def test_homogeneous_depth(sigma, per_voxel, nz):
    n, h = 64, 1.0 / 64
    sig = np.full((nz, 2, n), sigma, np.float32)
    alb = np.full(sig.shape, 0.5, np.float32)
    with gpu_grid(sig, alb, np.zeros(sig.shape, np.float32), h) as g:
        g.bake_directional((-1.0, 0.0, 0.0), 1.0, h / per_voxel)
        got = g.get_source()
    depth = float(sig[0, 0, 0]) * h * (n - np.arange(n) - 0.5)
    want = 0.5 * float(sig[0, 0, 0]) * np.exp(-depth)
    assert (np.abs(got - want) <= TOL * want).all()
