"""The FP64 helpers of the stage kernels return the bits of the plain expressions: the
quotient by a shared divisor, by a cell width (a power of two among them), and minmod; of
a zero the sign may differ as stated there.  Mantissas at random, near 1 and near 2, and exponents on both sides
of 2^-500 and 2^500, where the quotient changes form.  The expected values are numpy's."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")
from paper_2509_08971_gb300 import build  # noqa: E402

SOURCE = r"""
#include "hydro_math.cuh"
__global__ void ops(const double* a, const double* b, double* quot, double* width, double* mm, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    quot[i] = hh::div_by(a[i], b[i], __drcp_rn(b[i]), hh::mid_exponent(b[i]));
    width[i] = hh::sub_over_dx3(0.0, a[i], hh::make_width<double>(fabs(b[i])));
    mm[i] = hh::minmod(a[i], b[i]);
}
extern "C" int run(const double* a, const double* b, double* quot, double* width, double* mm, int n) {
    ops<<<(n + 255) / 256, 256>>>(a, b, quot, width, mm, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64_bits")
    (d / "ops.cu").write_text(SOURCE)
    out = d / "ops.so"
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "--fmad=false", "-shared", "-Xcompiler", "-fPIC",
                    "-I", build.CSRC, str(d / "ops.cu"), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))

    def run(a, b):
        dev = [torch.tensor(v, device="cuda") for v in (a, b)] + [torch.empty(len(a), dtype=torch.float64, device="cuda")
                                                                 for _ in range(3)]
        assert lib.run(*[ctypes.c_void_p(t.data_ptr()) for t in dev], len(a)) == 0
        return [t.cpu().numpy() for t in dev[2:]]

    return run


def _values(n, rng):
    """Mantissas of three kinds, exponents small, anywhere in the short form's range, and about its ends."""
    kind = rng.integers(0, 3, n)
    tail = rng.integers(0, 64, n) * 2.0 ** -52
    mant = np.where(kind == 0, 1.0 + rng.random(n), np.where(kind == 1, 1.0 + tail, 2.0 - 2.0 ** -52 - tail))
    at = rng.integers(0, 3, n)
    exp = np.where(at == 0, rng.integers(-3, 4, n),
                   np.where(at == 1, rng.integers(-500, 501, n), rng.choice([-500, 500], n) + rng.integers(-2, 3, n)))
    return np.ldexp(mant, exp) * rng.choice([-1.0, 1.0], n)


def _same(got, want):
    bad = np.flatnonzero(got.view(np.int64) != want.view(np.int64))
    return not len(bad), (len(bad), bad[:3], got[bad[:3]], want[bad[:3]])


def test_bits_of_the_plain_expressions(ops):
    rng = np.random.default_rng(23)
    n = 1 << 20
    a, b = _values(n, rng), _values(n, rng)
    a[:1000] = rng.choice([0.0, -0.0], 1000)
    b[1000:1500] = np.ldexp(1.0, rng.integers(-60, 61, 500))      # widths that are powers of two
    close = rng.integers(0, n, n // 8)
    a[close] = b[close] * rng.choice([1.0, -1.0, 1.0 + 2.0 ** -52, 1.0 - 2.0 ** -53], len(close))
    quot, width, _ = ops(a, b)
    with np.errstate(all="ignore"):
        quot, want = (np.where(v == 0.0, 0.0, v) for v in (quot, a / b))
        assert _same(quot, want)[0], _same(quot, want)[1]
        want = 0.0 - a / np.abs(b)
    assert _same(width, want)[0], _same(width, want)[1]


def test_minmod_bits(ops):
    rng = np.random.default_rng(29)
    n = 1 << 18
    a, b = _values(n, rng), _values(n, rng)
    special = np.array([0.0, -0.0, 5e-324, -5e-324, 1.0, -1.0, np.inf, -np.inf, np.nan, 2.0 ** -1022])
    a[:100], b[:100] = np.repeat(special, 10), np.tile(special, 10)
    _, _, got = ops(a, b)
    with np.errstate(all="ignore"):
        want = np.where((a > 0) & (b > 0), np.where(a <= b, a, b), np.where((a < 0) & (b < 0), np.where(-a <= -b, a, b), 0.0))
    got = np.where(got == 0.0, 0.0, got)
    assert _same(got, want)[0], _same(got, want)[1]
