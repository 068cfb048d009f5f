"""1D and 2D meshes of many strips: blocks of several warps, of which the last is short,
against the tile of one warp per block, bit for bit, with the rate and the totals that the
block combines."""
import numpy as np
import pytest

import oracle

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


# rows whose last cells share a warp between row chunks (remainders 1 .. 12 of 28), with and
# without full strips before them, beside remainders that do not; chunks that leave groups empty
@pytest.mark.parametrize("nx", [2, 3, 5, 6, 7, 12, 13, 28, 29, 32, 33, 40, 41, 57, 68, 69])
@pytest.mark.parametrize("ny", [2, 3, 17, 97])
@pytest.mark.parametrize("bc", [hh.HARD_BC_PERIODIC, hh.HARD_BC_OUTFLOW, hh.HARD_BC_REFLECT])
def test_rows_with_a_short_last_strip(nx, ny, bc):
    gam, shape = 1.4, (1, ny, nx)
    U0 = _state(shape, torch.float64).cpu().numpy()
    g = oracle.Grid(shape, gam, bc)
    ref, _, _ = g.run(U0, 2, 0.3)
    for dtype, tol in ((torch.float64, 1e-12), (torch.float32, 3e-6)):   # two steps of O(10) roundings
        base = None
        for tile in (-1, 0, 1, 2):
            m = hh.HardHydro(shape, gam, bc, dtype=dtype, tile=tile)
            U = torch.tensor(U0, dtype=dtype, device="cuda")
            t, dts, tot = m.advance(U, 2, 0.3, log_dt=True, log_totals=True)
            assert m.get_error() == hh.HARD_OK
            if base is None:
                base = (U, t, dts)
                for f in range(5):
                    big = max(np.abs(ref[f]).max(), 1e-3 * np.abs(ref).max())
                    assert np.abs(U[f].double().cpu().numpy() - ref[f]).max() <= tol * big, (dtype, f)
            assert all(torch.equal(a, b) for a, b in zip((U, t, dts), base)), (dtype, tile)
            assert np.allclose(tot[-1].cpu().numpy(), np.array(m.totals(U)), rtol=1e-10, atol=1e-10), (dtype, tile)
        # the same mesh among others of a batch
        B = hh.HardBatch([nx, 40, nx], [ny, 9, 1], gam, bc, dtype=dtype)
        P = B.pack([U0, _state((1, 9, 40), torch.float64).cpu(), _state((1, 1, nx), torch.float64).cpu()])
        t = B.step(P, 2, 0.3)
        # (a unit box of nx x ny cells, as above)
        assert torch.equal(B.view(P, 0), base[0]) and float(t[0]) == float(base[1]), dtype
