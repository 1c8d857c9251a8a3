"""The pointwise kernels' FP64 reciprocal and reciprocal square root (kernel header), compiled into
a small library, over every exponent and at the values that take the library functions."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_18221_gb300", "csrc")
SOURCE = r"""
#include "fp_convert.cuh"
__global__ void k(const double* x, double* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[4 * i] = gk::rcp64(x[i]);
    y[4 * i + 1] = gk::rsqrt64(x[i]);
    y[4 * i + 2] = 1.0 / x[i];
    y[4 * i + 3] = rsqrt(x[i]);
}
extern "C" int run(const double* x, double* y, int n) {
    k<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    torch = pytest.importorskip("torch")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("reciprocals")
    (d / "r.cu").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a", "-shared", "-Xcompiler",
                    "-fPIC", "-I" + CSRC, str(d / "r.cu"), "-o", str(d / "r.so")], check=True)
    torch.cuda.init()
    lib = ctypes.CDLL(str(d / "r.so"))

    def run(x):
        xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        yd = torch.empty(4 * xd.numel(), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(yd.data_ptr()), xd.numel()) == 0
        return yd.cpu().numpy().reshape(-1, 4).T
    return run


def _ulps(got, exact):
    """|got - exact| in units in the last place of the exact value."""
    err = np.abs(got.astype(np.longdouble) - exact)
    return float((err / np.spacing(np.abs(exact.astype(np.float64))).astype(np.longdouble)).max())


def test_every_exponent(evaluate):
    rng = np.random.default_rng(1)
    # fields 1 .. 2045: the reciprocals of all are normal numbers or the largest subnormals
    field = np.repeat(np.arange(1, 2046, dtype=np.uint64), 2000)
    mant = rng.integers(0, 2 ** 52, field.size, dtype=np.uint64)
    mant[::500], mant[1::500], mant[2::500] = 0, 2 ** 52 - 1, 2 ** 32 - 1
    x = ((field << np.uint64(52)) | mant).view(np.float64)
    rcp, rsq, div, lib = evaluate(x)
    one = np.longdouble(1)
    # the seeds read and keep 20 bits of mantissa: at most 2^-19 off, so what the third-order step
    # leaves out is at most 2^-57 of 1/x and (5/16) 2^-54 of 1/sqrt(x): 1/16 and 5/32 of the last place
    # on top of the final rounding
    assert _ulps(rcp, one / x.astype(np.longdouble)) <= 0.5 + 1 / 16 + 2.0 ** -8
    assert _ulps(rsq, one / np.sqrt(x.astype(np.longdouble))) <= 0.5 + 5 / 32 + 2.0 ** -8
    print("ulp: rcp %.4f (differs from 1/x: %.2e)  rsqrt %.4f (library %.4f)" % (
        _ulps(rcp, one / x.astype(np.longdouble)), np.mean(rcp != div),
        _ulps(rsq, one / np.sqrt(x.astype(np.longdouble))), _ulps(lib, one / np.sqrt(x.astype(np.longdouble)))))
    # odd in x, as the division is
    assert np.array_equal(evaluate(-x)[0], -rcp)


def test_values_outside_the_fast_range(evaluate):
    tiny = np.array([63, 64, 1982, 1983], dtype=np.uint64) << np.uint64(52)
    edge = np.concatenate([tiny.view(np.float64), (tiny | np.uint64(2 ** 52 - 1)).view(np.float64)])
    x = np.concatenate([[0.0, -0.0, 5e-324, -5e-324, 2.0 ** -1023, np.inf, -np.inf, np.nan, -1.0, -2.0 ** -1000,
                         -2.0 ** 1000, np.finfo(float).max], edge])
    rcp, rsq, div, lib = evaluate(x)
    np.testing.assert_array_equal(rcp[:12], div[:12])     # the division itself
    np.testing.assert_allclose(rcp[12:], div[12:], rtol=2.0 ** -52)
    assert np.array_equal(np.signbit(rcp[:2]), [False, True])
    np.testing.assert_allclose(rsq, lib, rtol=2.0 ** -52)
    assert np.isnan(rsq[[7, 8, 9, 10]]).all()
