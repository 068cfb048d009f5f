"""The diffusion's residual norm of a level stored by colour: with x = 0 and D = 0 the
residual is b, here one value everywhere, whose FP32 square rounds the same way addition
after addition."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
hh = pytest.importorskip("paper_2509_08971_gb300")
from paper_2509_08971_gb300 import build  # noqa: E402

SOURCE = r"""
#include "fld_split.cuh"
extern "C" int run(float* x, const float* b, const float* D, int n0, int n1, int n2, int stride, int chunk,
                   double* out) {
    hh::SplitArgs<float> a{};
    a.x = x; a.b = b; a.D = D;
    a.n[0] = n0; a.n[1] = n1; a.n[2] = n2;
    a.h = (n0 + 1) / 2;
    a.stride = stride;
    a.groups = (a.h + 3) / 4;
    a.color = n1 * n2 * stride;
    const dim3 grid((a.groups * n1 + 127) / 128, (n2 + chunk - 1) / chunk);
    for (int c = 0; c < 2; ++c)
        hh::split_norm_kernel<float, true><<<grid, 128>>>(a, c, chunk, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def norm(tmp_path_factory):
    d = tmp_path_factory.mktemp("fld_norm")
    (d / "norm.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC,
                    str(d / "norm.cu"), "-o", str(d / "norm.so")], check=True)
    return ctypes.CDLL(str(d / "norm.so")).run


@pytest.mark.parametrize("n", [(64, 64, 64), (61, 7, 33), (9, 130, 17)])
@pytest.mark.parametrize("chunk", [1, 8])
def test_sum_of_squares(norm, n, chunk):
    n0, n1, n2 = n
    stride = ((n0 + 1) // 2 + 3) // 4 * 4
    value = 1.0 + 2.0 ** -21
    x, D = (torch.zeros(2 * n2 * n1 * stride, device="cuda") for _ in range(2))
    b = torch.zeros((2, n2, n1, stride), device="cuda")
    for c in range(2):
        for s in range(2):                       # rows of parity s hold (n0 - s + 1) / 2 cells
            jk = (torch.arange(n2)[:, None] + torch.arange(n1)[None, :] + c) % 2 == s
            b[c][jk.cuda(), :(n0 - s + 1) // 2] = value
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    assert norm(ptr(x), ptr(b), ptr(D), n0, n1, n2, stride, chunk, ptr(out)) == 0
    want = n0 * n1 * n2 * np.float64(np.float32(value)) ** 2
    # seven FP32 additions of two vectors, each within 2^-24 of its sum; FP64 beyond
    assert abs(out.item() - want) <= 7 * 2.0 ** -24 * want, out.item() / want - 1
