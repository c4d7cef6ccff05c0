"""The FP64 form's quotient, reciprocal, root and comparison on the device, over the exponents in use and beyond.

From an approximation good to 2^-20, one Newton-Raphson or Goldschmidt step leaves 2^-39 at most; the quotient and the
root are then corrected by their exact remainders, which leaves the last rounding and 2^-70: within an ulp of the
correctly rounded value.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r"""
#include "rr_device.cuh"
__global__ void k(int which, const double* a, const double* b, double* out, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double x = a[i], y = b[i];
    out[i] = which == 0 ? rr::div64(x, y) : which == 1 ? rr::rcp64(x) : which == 2 ? rr::sqrt64(x) : rr::abs_le64(x, y);
}
extern "C" int run(int which, const double* a, const double* b, double* out, int n) {
    k<<<(n + 255) / 256, 256>>>(which, a, b, out, n);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2009_08500_gb300 import build as B
    d = tmp_path_factory.mktemp("arith")
    (d / "k.cu").write_text(SRC)
    root = os.path.dirname(B.HERE)
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-I", B.CSRC, "-I", os.path.join(root, "include"), "-o", str(d / "k.so"), str(d / "k.cu")], check=True)
    lib = ctypes.CDLL(str(d / "k.so"))

    def call(which, a, b):
        ta, tb = (torch.as_tensor(np.ascontiguousarray(v, np.float64), device="cuda") for v in np.broadcast_arrays(a, b))
        out = torch.empty_like(ta)
        assert lib.run(which, *(ctypes.c_void_p(t.data_ptr()) for t in (ta, tb, out)), ta.numel()) == 0
        return out.cpu().numpy()
    return call


def ulps(x, ref):
    return np.abs(x - ref) / np.spacing(np.abs(ref))


def spread(n, lo, hi, seed):
    rng = np.random.default_rng(seed)
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


def test_quotient_and_reciprocal(fn):
    n = 200_000
    a, b = spread(n, -200, 200, 1), spread(n, -200, 200, 2)
    a[: n // 2] *= -1.0
    b[::3] *= -1.0
    assert ulps(fn(0, a, b), a / b).max() <= 1.0
    near = 1.0 + np.arange(-500, 500) * 2.0 ** -52
    assert ulps(fn(0, 1.0, near), 1.0 / near).max() <= 1.0
    assert ulps(fn(0, near, near[::-1].copy()), near / near[::-1]).max() <= 1.0
    assert (fn(0, np.zeros(4), [1.0, -3.0, 1e100, 1e-100]) == 0).all()
    r = fn(1, b, 0.0)
    assert np.abs(r.astype(np.longdouble) * b - 1).max() <= 2.0 ** -39


def test_root(fn):
    h = np.concatenate([spread(200_000, -958, 1000, 3), spread(20_000, -60, 4, 4), 1.0 + np.arange(500) * 2.0 ** -52,
                        np.arange(1.0, 200.0) ** 2, [2.0 ** -958]])
    assert ulps(fn(2, h, 0.0), np.sqrt(h)).max() <= 1.0
    zero = np.array([0.0, -0.0, 2.0 ** -959, 2.0 ** -960, 1e-300, 5e-324, -1.0, -1e-200])
    assert (fn(2, zero, 0.0) == 0).all()


def test_comparison(fn):
    nan = np.array([0x7FF8000000000000, 0xFFF8000000000000, 0x7FFFFFFFFFFFFFFF, 0xFFFFFFFFFFFFFFFF], np.uint64).view(np.float64)
    x = np.concatenate([nan, [0.0, -0.0, 0.3, -0.3, 0.30000000000000004, np.inf, -np.inf, 1e-310, -1e300]])
    for y in (0.0, 0.3, 1e30, -1.0, np.inf, 1e-308):
        with np.errstate(invalid="ignore"):
            ref = np.abs(x) <= y
        assert np.array_equal(fn(3, x, y), ref.astype(np.float64))
