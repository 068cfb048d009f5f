"""Strip kernels of 1D and 2D meshes: 28 cells per warp, one, two, four or many
rows.  Sizes at the edges of strips and row chunks, every boundary kind: FP64
against the oracle, and every tile of both types equal bit for bit (the rows per
warp change no arithmetic)."""
import numpy as np
import pytest

import hydro_inputs as H
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")

SHAPES = [(1, 1, 2), (1, 1, 27), (1, 1, 28), (1, 1, 29), (1, 1, 113), (1, 2, 2), (1, 3, 30),
          (1, 5, 56), (1, 16, 57), (1, 17, 28), (1, 33, 85), (4, 1, 29), (18, 31, 1)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("bc", [0, 1, 2])
def test_strips(shape, bc):
    gam = 1.4
    U = H.smooth_3d(0, seed=5, gamma=gam, shape=shape)
    rng = np.random.default_rng(1)
    U[0] += 0.1 * rng.random(shape)
    g = oracle.Grid(shape, gam, bc)
    dt = 0.3 / g.max_rate(U)
    ref, _, _ = g.run(U, 3, 0.3)
    for dtype in (torch.float64, torch.float32):
        base = None
        m = hh.HardHydro(shape, gam, bc, dtype=dtype)
        for tile in range(-1, m.tile_count()):
            m.set_kernel(hh.HARD_KERNEL_FUSED, tile)
            Ud = torch.tensor(U, dtype=dtype, device="cuda")
            V = m.step(Ud, dt)
            t, _, tot = m.advance(Ud, 3, 0.3, log_totals=True)
            assert m.get_error() == hh.HARD_OK
            if base is None:
                base = (V, Ud, t)
                # FP32: three steps of O(10) roundings of the largest value
                tol = 1e-12 if dtype == torch.float64 else 3e-6
                for f in range(5):
                    big = max(np.abs(ref[f]).max(), 1e-3 * np.abs(ref).max())
                    err = np.abs(Ud[f].double().cpu().numpy() - ref[f]).max()
                    assert err <= tol * big, (dtype, f, err / big)
            assert all(torch.equal(a, b) for a, b in zip((V, Ud, t), base)), (dtype, tile)
            # the totals log against the state the last step left
            want = Ud.double().sum(dim=(1, 2, 3)) / np.prod(shape)
            assert torch.allclose(tot[-1], want, rtol=1e-6, atol=1e-6), (dtype, tile)
