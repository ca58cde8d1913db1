"""The FP64 helpers of the FP64-bound kernels, each by itself, against numpy in
units of the last place.  Bounds: the estimate's error of 2^-20 leaves 2^-60 after
the third-order step, so rcp64 rounds once after nearly exact terms (1 ulp);
rsqrt64 also rounds d y, worth half an ulp, before its last rounding (2);
exp_neg64 has the table entry's and the last rounding, numpy's own half (2)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1709_08070_gb300 import build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

SOURCE = """
#include "math64.cuh"
using namespace ibim;
__global__ void eval(int what, const double* x, double* y, long n, const double* tab)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = what == 0 ? rcp64(x[i]) : what == 1 ? rsqrt64(x[i]) : exp_neg64(x[i], tab);
}
extern "C" int run(int what, const double* x, double* y, long n, const double* tab)
{
    eval<<<(unsigned)((n + 255) / 256), 256>>>(what, x, y, n, tab);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def evaluate(tmp_path_factory):
    d = tmp_path_factory.mktemp("math64")
    src, out = str(d / "m.cu"), str(d / "m.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + build.CSRC,
                    "-I" + os.path.join(build.ROOT, "include"), src, "-o", out], check=True)
    fn = ctypes.CDLL(out).run
    p = ctypes.c_void_p
    fn.argtypes = [ctypes.c_int, p, p, ctypes.c_long, p]
    tab = torch.from_numpy(np.exp2(np.arange(512) / 512.0)).cuda()

    def call(what, x):
        a = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        y = torch.empty_like(a)
        assert fn(what, a.data_ptr(), y.data_ptr(), a.numel(), tab.data_ptr()) == 0
        return y.cpu().numpy()
    return call


def _ulps(got, want):
    return float(np.max(np.abs(got - want) / np.spacing(np.abs(want))))


def _arguments(lo, hi):
    rng = np.random.default_rng(2)
    m = np.concatenate([1.0 + rng.random(200000), 1.0 + np.arange(2048) / 2048.0, 2.0 - 2.0 ** -np.arange(1.0, 53.0)])
    return np.ldexp(m, rng.integers(lo, hi, m.size))


def test_reciprocal(evaluate):
    d = _arguments(-1000, 1000)
    assert _ulps(evaluate(0, d), 1.0 / d) <= 1.0


def test_reciprocal_square_root(evaluate):
    d = _arguments(-1000, 1000)
    want = (1.0 / np.sqrt(d.astype(np.longdouble))).astype(np.float64)
    assert _ulps(evaluate(1, d), want) <= 2.0


def test_exponential(evaluate):
    rng = np.random.default_rng(3)
    step = np.log(2.0) / 512.0
    edges = (np.arange(0, 40000)[:, None] + np.array([0.0, 0.5 - 1e-12, 0.5, 0.5 + 1e-12])).ravel() * step
    x = np.concatenate([[0.0, 5e-324, 1e-300, 1e-20, 1e-9], rng.uniform(0.0, 1e-3, 50000), rng.uniform(0.0, 699.0, 200000),
                        edges])
    assert _ulps(evaluate(2, x), np.exp(-x)) <= 2.0
    far = evaluate(2, np.array([700.0, 700.5, 745.0, 1e4, 1e308]))
    assert np.all((far > 0.0) & (far <= np.exp(-699.0)))
