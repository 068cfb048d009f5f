"""The second scheme in FP64 on states below 2^-500, whose quotients take the IEEE
division: its indicators are squares and underflow there, which leaves the linear weights."""
import numpy as np
import pytest

import hydro_inputs as H
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


@pytest.mark.parametrize("shape", [(1, 1, 70), (1, 9, 31), (7, 6, 34)])
@pytest.mark.parametrize("exponent", [-900, -502, -501, -500])
def test_weno_step_of_small_states(shape, exponent):
    gam = 1.4
    U = H.smooth_3d(0, seed=3, gamma=gam, shape=shape) * 2.0 ** exponent
    U[1, ..., ::3] = 0.0
    g = oracle.Grid(shape, gam, oracle.BC_OUTFLOW, scheme=hh.HARD_SCHEME_WENO5Z_HLL)
    dt = 0.3 / g.max_rate(U)
    ref = g.step(U, dt)
    assert np.isfinite(ref).all()
    m = hh.HardHydro(shape, gam, hh.HARD_BC_OUTFLOW, dtype=torch.float64, scheme=hh.HARD_SCHEME_WENO5Z_HLL)
    got = m.step(torch.tensor(U, device="cuda"), dt).cpu().numpy()
    # one step of O(30) roundings per term, as of states of order one
    for f in range(5):
        big = max(np.abs(ref[f]).max(), 1e-3 * np.abs(ref).max())
        assert np.abs(got[f] - ref[f]).max() <= 1e-12 * big, f
