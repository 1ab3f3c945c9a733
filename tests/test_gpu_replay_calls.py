"""fld_iterate's replays call by call, against calls too short to be replayed (counts
below four) on a grid of their own: changed counts, factors, sources, media and
states between the calls, every sweep family, a caller's stream and the legacy
stream."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

fld = pytest.importorskip("paper_1403_8105_gb300")
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

from test_gpu_parity import random_case  # noqa: E402


def same(g, ref, what):
    got, want = g.get_state(), ref.get_state()
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1]), what


@pytest.mark.parametrize("precision,bf16", [("fp32", 0), ("fp32", 1), ("pair", 0), ("pair", 1), ("mixed", 0)])
@pytest.mark.parametrize("legacy", [0, 1])
@pytest.mark.parametrize("shape", [(11, 14, 37), (40, 44, 42)])
def test_every_call_has_the_bits_of_launched_passes(precision, bf16, legacy, shape):
    nz, ny, nx = shape
    sig, alb, j, h = random_case(shape, 7)
    rng = np.random.default_rng(7)
    padded = tuple(n + 2 for n in shape)

    def par(omega, depth, limiter="lp"):
        return fld.params(precision=precision, omega=omega, warm_start=1, temporal_depth=depth, medium_bf16=bf16,
                          limiter=limiter)

    stream = torch.cuda.Stream()
    with fld.Grid(nx, ny, nz, h, stream=1 if legacy else stream.cuda_stream) as g, fld.Grid(nx, ny, nz, h) as ref:
        def both(f):
            f(g)
            f(ref)

        def call(n, omega, limiter="lp"):
            g.iterate(par(omega, 0, limiter), n)
            while n > 0:                               # passes launched one by one, whatever was called before
                ref.iterate(par(omega, -1, limiter), min(n, 3))
                n -= 3
            same(g, ref, (n, omega, limiter))

        both(lambda x: x.set_medium(sig, alb))
        both(lambda x: x.set_source(j))
        state = rng.uniform(0.05, 1.5, padded), rng.uniform(0.0, 0.1, padded)
        both(lambda x: x.set_state(*state))
        for n, omega in [(5, 1.4)] * 5 + [(6, 1.4)] * 4 + [(6, 1.2)] * 4 + [(5, 1.4)] * 4:
            call(n, omega)
        for k in range(4):                             # a new source, as a moved light, before every call
            both(lambda x: x.set_source((j * (1.0 + 0.1 * k)).astype(np.float32)))
            call(6, 1.4)
        both(lambda x: x.set_medium(0.5 * sig, alb))
        for _ in range(4):
            call(6, 1.4)
        both(lambda x: x.set_state(*state))
        for _ in range(2):
            call(6, 1.4)
        for _ in range(4):
            call(6, 1.4, "larsen")
