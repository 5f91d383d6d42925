"""The state reduction's reciprocal (rcp64.cuh) against exact arithmetic: within half a unit in the last place and 2^-10 of
one, over mantissas and exponents, and the library's division outside its range."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from tests.host_build import CSRC, cuda_home

pytestmark = pytest.mark.gpu

SOURCE = """
#include "rcp64.cuh"
__global__ void k(int n, const double* x, double* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = heat::rcp_or_0(x[i]);
}
extern "C" int rcp(int n, const double* x, double* y) {  // device buffers
    k<<<(n + 255) / 256, 256>>>(n, x, y);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def rcp(tmp_path_factory):
    import torch

    d = str(tmp_path_factory.mktemp("rcp"))
    src, so = os.path.join(d, "rcp.cu"), os.path.join(d, "librcp.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([os.path.join(cuda_home(), "bin", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                    "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def run(x):
        t = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        y = torch.empty_like(t)
        assert lib.rcp(t.numel(), ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(y.data_ptr())) == 0
        return y.cpu().numpy()

    return run


def _units_off(x, y):
    """|y - 1/x| in units of the last place of y, exactly."""
    return abs(Fraction(float(y)) - 1 / Fraction(float(x))) / Fraction(float(np.spacing(y)))


BOUND = Fraction(1, 2) + Fraction(1, 2**10)


def test_mantissas(rcp):
    rng = np.random.default_rng(1)
    top = np.arange(1 << 12) / 4096.0  # every leading 12 bits, with random and extreme tails
    ulp = 2.0**-52
    x = 1.0 + np.concatenate([top, top + 2.0**-12 - ulp, np.arange(40) * ulp, 1.0 - np.arange(1, 41) * ulp,
                              rng.random(20000)])
    y = rcp(x)
    # (at powers of two the neighbour below is half a unit away: 1/x is exact there)
    assert y[0] == 1.0
    assert max(_units_off(a, b) for a, b in zip(x, y)) <= BOUND


def test_exponents(rcp):
    e = np.arange(-1022, 1024)
    m = np.array([1.0, 1.0 + 2.0**-52, 1.3333333333333333, 1.5, 2.0 - 2.0**-52])
    x = np.ldexp(m[:, None], e[None, :]).ravel()
    y, normal = rcp(x), np.abs(1.0 / x) >= 2.0**-1022
    assert max(_units_off(a, b) for a, b in zip(x[normal], y[normal])) <= BOUND
    assert np.array_equal(y[~normal], 1.0 / x[~normal])


def test_outside_the_range(rcp):
    x = np.array([0.0, 5e-324, 2.0**-1030, 2.0**-1022, 2.0**1023, 1.7976931348623157e308, np.inf])
    with np.errstate(divide="ignore", over="ignore"):
        want = np.where(x > 0.0, 1.0 / np.where(x > 0.0, x, 1.0), 0.0)
    assert np.array_equal(rcp(x), want)
