"""FP64 stage parity over the exponent range: quotients by a shared divisor take
a short form inside 2^-500 .. 2^500 and an IEEE division outside it.  The Euler
equations are homogeneous in (rho, momentum, E), so a state scaled by a power
of two has the scaled result, bit for bit as long as nothing leaves the normal
range; the oracle's result is the check."""
import numpy as np
import pytest

import hydro_inputs as H
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


@pytest.mark.parametrize("shape", [(1, 1, 70), (1, 9, 31), (7, 6, 34)])
@pytest.mark.parametrize("exponent", [-900, -501, -499, 0, 499, 501, 900])
def test_scaled_state_matches_oracle(shape, exponent):
    gam = 1.4
    scale = 2.0 ** exponent
    U = H.smooth_3d(0, seed=3, gamma=gam, shape=shape) * scale
    U[1, ..., ::3] = 0.0                                # zero numerators
    for scheme in (hh.HARD_SCHEME_PLM_HLLC, hh.HARD_SCHEME_WENO5Z_HLL):
        g = oracle.Grid(shape, gam, oracle.BC_OUTFLOW, scheme=scheme)
        if scheme == hh.HARD_SCHEME_WENO5Z_HLL and not -499 <= exponent <= 0:
            continue        # its indicators square the state, and their ratio to 1e-30 overflows
        dt = 0.3 / g.max_rate(U)
        m = hh.HardHydro(shape, gam, hh.HARD_BC_OUTFLOW, dtype=torch.float64, scheme=scheme)
        got = m.step(torch.tensor(U, device="cuda"), dt).cpu().numpy()
        ref = g.step(U, dt)
        err = np.max(np.abs(got - ref), axis=(1, 2, 3))
        big = np.max(np.abs(ref), axis=(1, 2, 3))
        assert np.all(err <= 1e-12 * np.maximum(big, 1e-3 * big.max())), (exponent, err / big.max())
