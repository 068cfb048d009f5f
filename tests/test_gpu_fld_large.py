"""Diffusion on a mesh whose finest level exceeds 32-bit entries by colour (rows of nine
cells are padded to sixteen) while its cells do not: the levels below hold to the same
order.  The state is constant along z, so every plane is the solution of the 2D mesh."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


def test_finest_level_beyond_32_bit_entries_by_colour():
    nx, ny, nz = 9, 11600, 11600
    assert nx * ny * nz < 1 << 31 <= 16 * ny * nz
    if torch.cuda.mem_get_info()[0] < 80 << 30:
        pytest.skip("80 GB of device memory")
    g = torch.Generator(device="cuda").manual_seed(11)
    plane = torch.ones((5, 1, ny, nx), device="cuda")
    plane[0] += 0.5 * torch.rand((1, ny, nx), generator=g, device="cuda")
    E2 = 1.0 + 0.5 * torch.rand((1, ny, nx), generator=g, device="cuda")
    E3 = E2.expand(nz, ny, nx).contiguous()
    rtol = 1e-5
    sides = {"extent": (float(nx), float(ny), float(nz))}
    m2 = hh.HardHydro((1, ny, nx), 1.4, hh.HARD_BC_REFLECT, **sides)
    start = E2.clone()
    _, res2 = m2.fld_step(plane, E2, 30.0, 1.0, 1.0, rtol=rtol, max_cycles=40)
    m3 = hh.HardHydro((nz, ny, nx), 1.4, hh.HARD_BC_REFLECT, **sides)
    U = plane.expand(5, nz, ny, nx).contiguous()
    _, res3 = m3.fld_step(U, E3, 30.0, 1.0, 1.0, rtol=rtol, max_cycles=40)
    assert res2 <= rtol and res3 <= rtol, (res2, res3)
    # the smallest eigenvalue of the system is 1: each solution is within its residual of
    # the exact one, the FP32 residual within its rounding (diag x, ~50 x 6e-8)
    err = sum(float((E3[k:k + 400].double() - E2[0].double()).square().sum()) for k in range(0, nz, 400))
    norm = nz * float(start.double().square().sum())
    assert err <= (2 * (rtol + 3e-6)) ** 2 * norm, (err / norm) ** 0.5
