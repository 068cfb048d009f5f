"""Diffusion on meshes with levels above the one-block set: levels stored by
colour (rows of every remainder of a vector, wrapped and walled, axes that
coarsen and axes that do not, one to three dimensions) and levels in mesh order
(odd periodic axes), against the oracle's direct solve."""
import numpy as np
import pytest

from oracle import fld as OF

torch = pytest.importorskip("torch")
pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")

from test_gpu_fld import C, KAPPA, _dx, _state  # noqa: E402

CASES = [((1, 1, 8192), 0), ((1, 1, 5001), 1), ((1, 70, 68), 0), ((1, 75, 66), 2), ((20, 18, 34), 0),
         ((20, 18, 34), 1), ((16, 20, 50), 0), ((16, 22, 26), 0), ((20, 24, 12), 0), ((24, 22, 27), 2),
         ((26, 25, 30), 1), ((19, 21, 23), 1), ((17, 16, 48), 0), ((18, 20, 45), 0), ((30, 40, 8), 2),
         ((40, 30, 6), 0)]


@pytest.mark.parametrize("shape,bc", CASES)
def test_fld_levels(shape, bc):
    U, E = _state(shape, seed=sum(shape) + bc)
    U, E = (a.astype(np.float32).astype(np.float64) for a in (U, E))
    dx = _dx(shape)
    dt = 3.0 * min(d for d, n in zip(dx, shape[::-1]) if n > 1) ** 2 * 3
    ref = OF.fld_step(U[0], E, dt, C, KAPPA, dx, [bc] * 6)
    # the smallest eigenvalue of A is 1: the error is at most the residual;
    # FP32 residuals bottom out at the rounding of diag x, ~20 x 6e-8
    for dtype, rtol, tol in ((torch.float64, 1e-12, 1e-10), (torch.float32, 1e-5, 1e-5)):
        m = hh.HardHydro(shape, 1.4, bc, dtype=dtype, extent=(1.0, 0.8, 1.2))
        Ud = torch.tensor(U, dtype=dtype, device="cuda")
        first = torch.tensor(E, dtype=dtype, device="cuda")
        cyc, res = m.fld_step(Ud, first, dt, C, KAPPA, rtol=rtol, max_cycles=200)
        assert res <= rtol, (dtype, cyc, res)
        err = np.linalg.norm(first.double().cpu().numpy() - ref) / np.linalg.norm(ref)
        assert err <= tol, (dtype, err)
        # the handle's arrays hold nothing of one call for the next
        again = torch.tensor(E, dtype=dtype, device="cuda")
        other = 2.0 + again.flip(0)
        m.fld_step(Ud, other, dt, C, KAPPA, rtol=rtol, max_cycles=3)
        cyc2, _ = m.fld_step(Ud, again, dt, C, KAPPA, rtol=rtol, max_cycles=200)
        err = float((again.double() - first.double()).norm() / first.double().norm())
        assert cyc2 == cyc and err <= tol, (dtype, cyc, cyc2, err)
