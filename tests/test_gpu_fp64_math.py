"""The FP64 functions that the sums and the FP64 cycle call in place of CUDA's, over their whole
argument range, against extended precision.  The bounds add up the roundings of each method."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "fp64_math.cuh"
using namespace pbg;
__global__ void k(int which, const double *x, double *y, int n) {
    __shared__ double tab[64];
    if (threadIdx.x < 64) tab[threadIdx.x] = exp2((double)threadIdx.x * 0.015625);
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) y[i] = %s;
}
extern "C" int run(int which, const double *x, double *y, int n) {
    k<<<(n + 255) / 256, 256>>>(which, x, y, n);
    return (int)cudaDeviceSynchronize();
}
"""
FUNCTIONS = ["exp_neg_fp64(x[i], tab)", "rsqrt_fp64(x[i])", "rcp_fp64(x[i])"]


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_09323_gb300 import build
    d = tmp_path_factory.mktemp("fp64")
    chain = "".join(f"which == {q} ? {f} : " for q, f in enumerate(FUNCTIONS)) + "0.0"
    (d / "t.cu").write_text(SOURCE % chain)
    subprocess.run([build.nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, "-shared", "-Xcompiler", "-fPIC",
                    "-o", str(d / "t.so"), str(d / "t.cu")], check=True)
    lib = ctypes.CDLL(os.fspath(d / "t.so"))

    def f(which, x):
        xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        y = torch.empty_like(xd)
        torch.cuda.synchronize()
        assert lib.run(which, ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(y.data_ptr()), len(x)) == 0
        return y.cpu().numpy()

    return f


def test_exp_neg(call):
    rng = np.random.default_rng(1)
    step = np.log(2.0) / 64
    edges = (np.arange(65400) + 0.5) * step  # where n changes
    u = np.concatenate([[0.0, 5e-324, 1e-300, 707.999], np.exp(rng.uniform(-40, np.log(707.9), 200000)),
                        rng.uniform(0, 707.9, 200000), np.arange(65400) * step, edges, np.nextafter(edges, 0),
                        np.nextafter(edges, 1000)])
    u = u[u < 708.0]
    y = call(0, u)
    exact = np.exp(-u.astype(np.longdouble))
    # in units of 2^-53: the polynomial's last step 1 and its remainder 0.4, the table (exp2, good to one
    # unit in the last place) 2, the product 1
    assert np.abs(y / exact - 1).max() <= 4.5 * 2.0 ** -53
    # underflow, up to the largest arguments
    big = np.concatenate([[708.0, 1e3, 2.3e7, np.inf, 1.7e308], 2.0 ** np.arange(10, 1024),
                          np.exp(rng.uniform(np.log(708.1), 700, 100000)), 2.33e7 * np.arange(1, 200)])
    assert np.all(call(0, big) == 0.0)


def test_rsqrt(call):
    rng = np.random.default_rng(2)
    m = np.concatenate([1.0 + rng.random(300000), 1.0 + np.arange(1 << 20) * 2.0 ** -20, np.nextafter([1.0, 2.0], 3.0)])
    a = np.concatenate([m, np.ldexp(m, rng.integers(-1022, 1023, len(m))), 2.0 ** np.arange(-1022, 1024),
                        [np.finfo(float).max, np.finfo(float).tiny]])
    exact = 1 / np.sqrt(a.astype(np.longdouble))
    # in units of 2^-53: the last step 1, e (one rounding of a y, halved by the series) 0.5, the remainder
    # 5/16 e^3, e up to 2^-18, 0.2
    assert np.abs(call(1, a) / exact - 1).max() <= 1.75 * 2.0 ** -53
    s = np.concatenate([[5e-324, np.nextafter(np.finfo(float).tiny, 0)], rng.integers(1, 1 << 52, 1000) * 5e-324])
    # subnormal: CUDA's function, good to two units
    assert np.abs(call(1, s) * np.sqrt(s.astype(np.longdouble)) - 1).max() <= 4 * 2.0 ** -53
    assert call(1, np.array([0.0, np.inf])).tolist() == [np.inf, 0.0]


def test_rcp(call):
    rng = np.random.default_rng(3)
    m = np.concatenate([1.0 + rng.random(300000), 1.0 + np.arange(1 << 20) * 2.0 ** -20, np.nextafter([1.0, 2.0], 3.0)])
    b = np.concatenate([m, np.ldexp(m, rng.integers(-1000, 1000, len(m))), 2.0 ** np.arange(-1000, 1001)])
    exact = 1 / b.astype(np.longdouble)
    # in units of 2^-53: the last step 1, e and e^2 2^-18 of that, the remainder e^3 (e up to 2^-18.5) 0.2
    assert np.abs(call(2, b) / exact - 1).max() <= 1.25 * 2.0 ** -53
