"""exp64 and rcp64 (csrc/xc_exp64.cuh) on the device against the host's long double."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1801_09803_gb300 import build as b

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

KERNEL = r"""
#include "xc_exp64.cuh"
__global__ void k(const double *x, double *e, double *r, int n) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    e[i] = xc::exp64(x[i]);
    r[i] = xc::rcp64(x[i]);
}
extern "C" int run(const double *x, double *e, double *r, int n) {
    k<<<(n + 255) / 256, 256>>>(x, e, r, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("prim")
    (d / "k.cu").write_text(KERNEL)
    subprocess.run([b.nvcc(), *b.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", b.CSRC,
                    "--expt-relaxed-constexpr", str(d / "k.cu"), "-o", str(d / "k.so")], check=True)
    L = C.CDLL(str(d / "k.so"))
    L.run.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]

    def f(x):
        t = torch.as_tensor(np.ascontiguousarray(x), device="cuda:0")
        e, r = torch.empty_like(t), torch.empty_like(t)
        torch.cuda.synchronize()
        assert L.run(t.data_ptr(), e.data_ptr(), r.data_ptr(), len(t)) == 0
        return e.cpu().numpy(), r.cpu().numpy()
    return f


def test_exp64(run):
    rng = np.random.default_rng(2)
    x = np.concatenate([np.arange(-5120, 5120) * (np.log(2.0) / 1024), rng.uniform(-707.99, 707.99, 200_000),
                        -10.0 ** rng.uniform(-300, 2.8, 20_000), [0.0, -0.0, 707.99999, -707.99999]])
    ref = np.exp(x.astype(np.longdouble))
    err = np.abs(run(x)[0].astype(np.longdouble) - ref) / np.spacing(ref.astype(np.float64))
    assert float(err.max()) < 0.51 + 2.0 ** -9   # the long double's own error included
    # the library's exponential beyond: limits, infinities, NaN
    e = run(np.array([708.5, -708.5, -745.0, -746.0, 709.9, np.inf, -np.inf, np.nan]))[0]
    assert np.all(np.isfinite(e[:3])) and e[3] == 0.0 and np.isposinf(e[4:6]).all() and e[6] == 0.0 and np.isnan(e[7])
    assert abs(e[0] / np.exp(708.5) - 1) < 1e-15 and abs(e[1] / np.exp(-708.5) - 1) < 1e-13


def test_rcp64(run):
    """Over the exponents of products of four quadratics: a last-place error."""
    rng = np.random.default_rng(3)
    x = rng.uniform(1.0, 2.0, 400_000) * 2.0 ** rng.integers(-990, 990, 400_000)
    r = run(x)[1]
    ref = 1 / x.astype(np.longdouble)
    assert float((np.abs(r.astype(np.longdouble) - ref) / np.spacing(ref.astype(np.float64))).max()) <= 1.0
    assert np.array_equal(run(-x[:1000])[1], -r[:1000])
