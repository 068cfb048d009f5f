"""The launch rules' choices (tile -1) on meshes about the lines that measurements drew;
host code only."""
import pytest

torch = pytest.importorskip("torch")
import paper_2509_08971_gb300 as hh  # noqa: E402
from paper_2509_08971_gb300 import build  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def _tile(shape, dtype=torch.float32, kernel=hh.HARD_KERNEL_FUSED):
    return tuple(hh.HardHydro(shape, 1.4, hh.HARD_BC_PERIODIC, dtype=dtype, kernel=kernel).tile_info(-1))


def test_1d_warps_per_block():
    for n in (2, 400, 16000):
        assert _tile((1, 1, n)) == (32, 1, 1, 32)
    for shape in ((1, 1, 32000), (1, 10 ** 6, 1), (10 ** 7, 1, 1)):
        assert _tile(shape) == (32, 8, 1, 256)
        assert _tile(shape, torch.float64) == (32, 1, 1, 32)
