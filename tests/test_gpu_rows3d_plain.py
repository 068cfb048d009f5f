"""The plain 3D kernel at the launch rule's tile and chunk: the bits of the fixed tiles, at
sizes about the edges of 4- and 8-row tiles and of short chunks."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 4, 5), (7, 5, 33), (33, 9, 40), (20, 31, 64), (64, 64, 64), (5, 150, 150)])
@pytest.mark.parametrize("bc", [0, 1, 2])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_plain_tiles(shape, bc, dtype):
    g = torch.Generator(device="cuda").manual_seed(31)
    U0 = 0.1 * torch.rand((5,) + shape, generator=g, dtype=torch.float64, device="cuda")
    U0[0] += 1.0
    U0[4] += 2.5
    base = None
    for tile in (0, 1, 4, -1):
        m = hh.HardHydro(shape, 1.4, bc, dtype=dtype, kernel=hh.HARD_KERNEL_PLAIN, tile=tile)
        U = U0.to(dtype, copy=True)
        t, dts, tot = m.advance(U, 2, 0.3, log_dt=True, log_totals=True)
        assert m.get_error() == hh.HARD_OK
        want = torch.tensor(m.totals(U), dtype=torch.float64)
        assert torch.allclose(tot[-1].cpu(), want, rtol=1e-10, atol=1e-10), tile
        if base is None:
            base = (U, t, dts)
        assert all(torch.equal(a, b) for a, b in zip((U, t, dts), base)), tile
