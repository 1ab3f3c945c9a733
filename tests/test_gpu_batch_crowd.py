"""Batches large enough that their grids are in one another's way and run other
launch forms than alone: the bits stay those of the solo solves."""
import numpy as np
import pytest

import fld_inputs

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)


def grid(n, seed):
    sig, alb = fld_inputs.cloud_medium(n, seed=seed, albedo=0.95)
    g = fld.Grid(n, n, n, 1.0 / n)
    g.set_medium(sig, alb)
    g.bake_directional((0.0, 0.0, -1.0), 1.0)
    return g


# two grids (both run as alone); four, above which whole iterations per launch give way;
# four of 6100 voxels per SM of 152, above the line of the one-unknown passes; a batch
# crosses both lines as its grids finish
@pytest.mark.parametrize("edges", [(24, 20), (32, 24, 28, 20), (64, 50, 66, 64)])
@pytest.mark.parametrize("precision,kw", [("fp32", {}), ("pair", {}), ("mixed", dict(fp32_switch=1e9)),
                                          ("mixed", dict(anderson=4))])
def test_crowded_batches_equal_solo_solves(edges, precision, kw):
    p = fld.params(precision=precision, tol=2e-4, max_iters=640, check_every=64, **kw)
    want = []
    for a, n in enumerate(edges):
        with grid(n, a) as g:
            r = g.solve(p, check=False)
            want.append((r.iterations, g.get_state()))
    grids = [grid(n, a) for a, n in enumerate(edges)]
    try:
        _, rs = fld.fld_solve_batch(grids, p, check=False)
        for g, r, (its, state) in zip(grids, rs, want):
            assert r.iterations == its
            got = g.get_state()
            assert np.array_equal(got[0], state[0]) and np.array_equal(got[1], state[1])
    finally:
        for g in grids:
            g.close()
