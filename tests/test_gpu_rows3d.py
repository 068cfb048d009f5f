"""3D meshes whose rows are no multiple of 16 bytes (FP32: the warp-specialised
kernel fed by 4-byte copies), and the chunk lengths the launch rules choose:
sizes at the edges of tiles and chunks, every boundary kind, against the oracle;
the rule's tile, every fixed tile and any chunk give the same bits."""
import numpy as np
import pytest

import hydro_inputs as H
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")


def _state(shape, gam):
    U = H.smooth_3d(0, seed=7, gamma=gam, shape=shape)
    U[0] += 0.1 * np.random.default_rng(2).random(shape)
    return U


def _check(Ud, ref, tol, what):
    for f in range(5):
        big = max(np.abs(ref[f]).max(), 1e-3 * np.abs(ref).max())
        err = np.abs(Ud[f].double().cpu().numpy() - ref[f]).max()
        assert err <= tol * big, (what, f, err / big)


@pytest.mark.parametrize("shape", [(2, 2, 2), (3, 2, 3), (2, 3, 5), (5, 17, 31), (4, 15, 33), (7, 16, 34),
                                   (35, 9, 63), (3, 33, 65), (66, 5, 30), (41, 37, 53)])
@pytest.mark.parametrize("bc", [0, 1, 2, [2, 1, 0, 0, 1, 2]])
def test_rows_of_any_length(shape, bc):
    gam = 1.4
    U = _state(shape, gam)
    ref, _, _ = oracle.Grid(shape, gam, bc).run(U, 3, 0.3)
    for dtype, tol in ((torch.float64, 1e-12), (torch.float32, 3e-6)):   # 3 steps of O(10) roundings
        base = None
        m = hh.HardHydro(shape, gam, bc, dtype=dtype)
        # FP32's 64-wide tile runs the plain kernel, which rounds differently
        tiles = [t for t in range(m.tile_count()) if m.tile_info(t)[0] == 32]
        for tile in [-1] + tiles:
            m.set_kernel(hh.HARD_KERNEL_FUSED, tile)
            Ud = torch.tensor(U, dtype=dtype, device="cuda")
            t, _, tot = m.advance(Ud, 3, 0.3, log_totals=True)
            assert m.get_error() == hh.HARD_OK
            if base is None:
                base = (Ud, t)
                _check(Ud, ref, tol, dtype)
            assert torch.equal(Ud, base[0]) and torch.equal(t, base[1]), (dtype, tile)
            want = Ud.double().sum(dim=(1, 2, 3)) / np.prod(shape)
            assert torch.allclose(tot[-1], want, rtol=1e-6, atol=1e-6), (dtype, tile)


# rows at the edges of the x sweeps' segments (62 and 94 cells), columns that are
# no multiple of a block, rows shared by blocks, one and several chunks
SWEEPS = [(3, 3, 3), (4, 5, 127), (9, 3, 43), (30, 6, 130), (75, 7, 20), (3, 4, 62), (3, 5, 63), (4, 3, 94),
          (3, 3, 95), (3, 4, 187), (3, 3, 189)]


@pytest.mark.parametrize("shape", SWEEPS)
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_advect_sweeps(shape, bc):
    gam = 1.4
    U = _state(shape, gam)
    E = 1.0 + 0.5 * np.random.default_rng(4).random(shape)
    g = oracle.Grid(shape, gam, bc)
    dt = 0.3 / g.max_rate(U)
    ref = g.advect_E(U, E, dt)
    for dtype, tol in ((torch.float64, 1e-12), (torch.float32, 3e-6)):   # one step of O(30) roundings
        m = hh.HardHydro(shape, gam, bc, dtype=dtype)
        Ed = torch.tensor(E, dtype=dtype, device="cuda")
        m.advect_E(torch.tensor(U, dtype=dtype, device="cuda"), Ed, dt)
        assert np.abs(Ed.double().cpu().numpy() - ref).max() <= tol * np.abs(ref).max(), dtype


@pytest.mark.parametrize("shape", SWEEPS)
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_weno_sweeps(shape, bc):
    gam = 1.4
    U = _state(shape, gam)
    ref, _, _ = oracle.Grid(shape, gam, bc, scheme=1).run(U, 2, 0.3)
    for dtype, tol in ((torch.float64, 1e-12), (torch.float32, 6e-6)):   # 2 steps of O(30) roundings
        m = hh.HardHydro(shape, gam, bc, dtype=dtype, scheme=hh.HARD_SCHEME_WENO5Z_HLL)
        Ud = torch.tensor(U, dtype=dtype, device="cuda")
        _, _, tot = m.advance(Ud, 2, 0.3, log_totals=True)
        assert m.get_error() == hh.HARD_OK
        _check(Ud, ref, tol, dtype)
        want = Ud.double().sum(dim=(1, 2, 3)) / np.prod(shape)
        assert torch.allclose(tot[-1], want, rtol=1e-6, atol=1e-6), dtype
