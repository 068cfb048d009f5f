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


def test_3d_tiles():
    plain = {"kernel": hh.HARD_KERNEL_PLAIN}
    # meshes of a few planes: 8 rows cost less per block; deep ones: 16 cost less per plane
    for nz in (4, 5, 8):
        assert _tile((nz, 1000, 1000))[:2] == (32, 8)
    for n in (64, 128, 256, 512):
        assert _tile((n, n, n))[:2] == (32, 16)
        assert _tile((n, n, n), **plain)[:2] == (32, 4)
    # rows that TMA does not take
    assert _tile((93, 117, 150)) == (32, 8, 24, 256)
    assert _tile((4, 601, 499))[:2] == (32, 16)
    # beyond the rows that a grid of 8-row tiles takes nothing is chosen in its place
    assert _tile((2, 8 * 65535 + 1, 2)) == _tile((2, 8 * 65535 + 1, 2), **plain) == (32, 8, 32, 256)
