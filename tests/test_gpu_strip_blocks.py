"""1D and 2D meshes of many strips: blocks of several warps, of which the last is short,
against the tile of one warp per block, bit for bit, with the rate and the totals that the
block combines."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


def _state(shape, dtype):
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    U = 0.1 * torch.rand((5,) + shape, generator=g, dtype=torch.float64, device="cuda")
    U[0] += 1.0
    U[4] += 2.5
    U[1, ..., shape[2] // 3] += 0.7                  # the largest rate at one place
    return U.to(dtype)


@pytest.mark.parametrize("shape", [(1, 1, 21280), (1, 1, 21281 + 28 * 5), (1, 1, 100003), (1, 30001, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_1d_blocks(shape, dtype):
    base = None
    for tile in (0, 1, -1):
        m = hh.HardHydro(shape, 1.4, hh.HARD_BC_REFLECT, dtype=dtype, tile=tile)
        U = _state(shape, dtype)
        t, dts, tot = m.advance(U, 3, 0.3, log_dt=True, log_totals=True)
        assert m.get_error() == hh.HARD_OK
        if base is None:
            base = (U, t, dts)
        assert all(torch.equal(a, b) for a, b in zip((U, t, dts), base)), tile
        want = np.array(m.totals(U))
        assert np.allclose(tot[-1].cpu().numpy(), want, rtol=1e-12, atol=1e-12), tile
