"""The residual's sums over tens of millions of unknowns: equal terms, whose
roundings do not cancel, and terms of eight orders of magnitude."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

# the warps' sums and the CTAs' in FP64 (some thirty additions of 1.1e-16 at
# most along one path), a square root and a quotient
TOL = 4e-15
SOURCE = np.float32(0.456407607)


def relative_residual(n, source, precision):
    """Rbar / jbar where phi is 1 throughout, sigma' = source - 1/4 and albedo 0: the
    residual is exactly 1/4 everywhere."""
    medium = (source - np.float32(0.25)).astype(np.float32)
    with fld.Grid(n, n, n, 1.0) as g:
        dev = torch.device("cuda", 0)
        expand = [torch.from_numpy(np.ascontiguousarray(a.astype(np.float32))).to(dev)[:, None, None]
                  .expand(n, n, n).contiguous() for a in (medium, 0 * source, source)]
        g.set_medium(expand[0], expand[1])
        g.set_source(expand[2])
        one = torch.ones((n + 2,) * 3, dtype=torch.float64, device=dev)
        g.set_state(one, one)
        if precision is None:
            return g.residual(fld.params(precision="mixed"))
        p = fld.params(precision=precision, warm_start=1, max_iters=0, tol=0.0)
        return g.solve(p, check=False).rel_residual


@pytest.mark.parametrize("precision", [None, "fp32"])
@pytest.mark.parametrize("n", [9, 384])
def test_equal_terms(n, precision):
    got = relative_residual(n, np.full(n, SOURCE), precision)
    assert abs(got - 0.25 / float(SOURCE)) <= TOL * got


@pytest.mark.parametrize("n", [61, 200])
def test_spread_terms(n):
    source = np.geomspace(0.26, 2600.0, n).astype(np.float32)
    want = 0.25 / math.sqrt(math.fsum(float(s) ** 2 for s in source) / n)
    got = relative_residual(n, source, None)
    assert abs(got - want) <= TOL * want
