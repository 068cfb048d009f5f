"""The totals that the time loop logs from an FP32 state are as good as an FP64 sum,
however many cells a lane completes: against the standalone totals (FP64 from the first
addition) on near-uniform states, whose FP32 partial sums round the same way cell after
cell."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")

# A lane completes at most 72 cells.  With u = 2^-24 each addition's error is at most u times the
# sum so far, n u S after n cells, and enters the error word with another rounding: 2 n^2 u^2 S.
TOL = 2 * 72 ** 2 * 2.0 ** -48

CASES = [((1, 1, 3000), {}), ((1, 2000, 260), {}), ((1, 2000, 260), {"tile": 2}), ((1, 300, 300), {}),
         ((150, 64, 64), {}), ((150, 64, 64), {"tile": 1}), ((144, 40, 64), {"tile": 2}), ((150, 33, 35), {}),
         ((150, 33, 35), {"tile": 4}), ((150, 33, 64), {"kernel": hh.HARD_KERNEL_PLAIN, "tile": 3}),
         ((150, 20, 33), {"scheme": hh.HARD_SCHEME_WENO5Z_HLL}),
         ((1, 64, 64), {"scheme": hh.HARD_SCHEME_WENO5Z_HLL})]


@pytest.mark.parametrize("shape,kw", CASES)
@pytest.mark.parametrize("noise", [0.0, 1e-4])
def test_logged_totals_are_fp64_sums(shape, kw, noise):
    g = torch.Generator(device="cuda").manual_seed(17)
    U = torch.rand((5,) + shape, generator=g, device="cuda") * noise
    for f, v in enumerate((1.1, 0.37, -0.23, 0.11, 6.3)):
        U[f] += v
    m = hh.HardHydro(shape, 1.4, hh.HARD_BC_PERIODIC, dtype=torch.float32, **kw)
    _, _, log = m.advance(U, 2, 0.3, log_totals=True)
    assert m.get_error() == hh.HARD_OK
    want = np.array(m.totals(U))
    err = np.abs(log[-1].cpu().numpy() - want)
    assert np.all(err <= TOL * np.abs(want)), err / np.abs(want)
