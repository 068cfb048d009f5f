"""Diffusion on meshes with levels above the one-block set: levels stored by
colour (rows of every remainder of a vector, wrapped and walled, axes that
coarsen and axes that do not, one to three dimensions) and levels in mesh order
(odd periodic axes, small levels), against the oracle's linear system."""
import numpy as np
import pytest

from oracle import fld as OF

torch = pytest.importorskip("torch")
pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")

from test_gpu_fld import C, KAPPA, _dx, _state  # noqa: E402

CASES = [((1, 1, 140000), 0), ((1, 1, 131075), 1), ((1, 362, 370), 0), ((1, 365, 366), 2), ((52, 50, 52), 0),
         ((52, 50, 58), 1), ((44, 58, 54), 0), ((51, 53, 50), 2), ((50, 52, 55), 2), ((53, 49, 51), 1),
         ((64, 64, 34), 0), ((70, 90, 22), 2), ((130, 128, 8), 0), ((51, 60, 48), 0), ((20, 18, 34), 1),
         ((24, 22, 27), 2), ((19, 21, 23), 1), ((17, 16, 48), 0)]


@pytest.mark.parametrize("shape,bc", CASES)
def test_fld_levels(shape, bc):
    U, E = _state(shape, seed=sum(shape) + bc)
    U, E = (a.astype(np.float32).astype(np.float64) for a in (U, E))
    dx = _dx(shape)
    dt = 3.0 * min(d for d, n in zip(dx, shape[::-1]) if n > 1) ** 2 * 3
    D = OF.diffusion_coefficient(U[0], E, C, KAPPA, dx, [bc] * 6)
    A = OF.fld_matrix(D, dt, dx, [bc] * 6)
    ref = None
    # the smallest eigenvalue of A is 1: the error is at most the residual;
    # FP32 residuals bottom out at the rounding of diag x, ~20 x 6e-8
    for dtype, rtol, tol in ((torch.float64, 1e-12, 1e-10), (torch.float32, 1e-5, 2e-5)):
        m = hh.HardHydro(shape, 1.4, bc, dtype=dtype, extent=(1.0, 0.8, 1.2))
        Ud = torch.tensor(U, dtype=dtype, device="cuda")
        first = torch.tensor(E, dtype=dtype, device="cuda")
        cyc, res = m.fld_step(Ud, first, dt, C, KAPPA, rtol=rtol, max_cycles=200)
        assert res <= rtol, (dtype, cyc, res)
        got = first.double().cpu().numpy().ravel()
        if ref is None:
            err = np.linalg.norm(A @ got - E.ravel()) / np.linalg.norm(E)
            ref = got
        else:
            err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
        assert err <= tol, (dtype, err)
        # the handle's arrays hold nothing of one call for the next
        again = torch.tensor(E, dtype=dtype, device="cuda")
        other = 2.0 + again.flip(0)
        m.fld_step(Ud, other, dt, C, KAPPA, rtol=rtol, max_cycles=3)
        cyc2, _ = m.fld_step(Ud, again, dt, C, KAPPA, rtol=rtol, max_cycles=200)
        err = float((again.double() - first.double()).norm() / first.double().norm())
        assert cyc2 == cyc and err <= tol, (dtype, cyc, cyc2, err)
        # no half-sweep reads what it writes, unless a periodic axis is odd
        if bc != 0 or all(n == 1 or n % 2 == 0 for n in shape):
            assert torch.equal(again, first), dtype
