"""The FP64 reciprocal of the pair kernels (common.cuh) against the correctly rounded quotient.

The iteration's remainder is below 2^-60 and its last operation rounds once: the result is one of the
two numbers next to 1/x, so within one unit in the last place of the rounded quotient, over the range
that the comment states; zero, infinities and NaN as the divide gives them."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2208_14639_gb300 import build, vv10

pytestmark = pytest.mark.gpu

SOURCE = """
#include "common.cuh"
__global__ void k(const double* x, double* y, int n) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) y[i] = vv10::recip(x[i]);
}
extern "C" int run(const double* x, double* y, int n) {
    k<<<(n + 255) / 256, 256>>>(x, y, n);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def recip(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    d = tmp_path_factory.mktemp("recip")
    src, lib = os.path.join(d, "recip.cu"), os.path.join(d, "librecip.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-shared", "-cudart", "static", "-o", lib, src], check=True)
    run = ctypes.CDLL(lib).run

    def call(x):
        t = torch.from_numpy(x).to("cuda:0")
        y = torch.empty_like(t)
        torch.cuda.synchronize()
        assert run(ctypes.c_void_p(t.data_ptr()), ctypes.c_void_p(y.data_ptr()), len(x)) == 0
        return y.cpu().numpy()

    return call


def test_within_one_ulp(recip):
    rng = np.random.default_rng(0)
    n = 1 << 20
    x = np.concatenate([rng.uniform(1.0, 2.0, n), np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-1022, 1022, n)),
                        np.nextafter(2.0, 0.0) * np.ones(1), np.ldexp(np.ones(2044), np.arange(-1022, 1022))])
    x *= np.where(rng.integers(0, 2, len(x)) == 0, -1.0, 1.0)
    y = recip(x)
    assert (np.abs(y.view(np.int64) - (1.0 / x).view(np.int64)) <= 1).all()


def test_ends(recip):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0**1023])
    y = recip(x)
    with np.errstate(divide="ignore"):
        ref = 1.0 / x[:5]
    assert np.array_equal(y[:5], ref, equal_nan=True) and np.array_equal(np.signbit(y[:4]), np.signbit(ref[:4]))
    assert y[5] == 0.0
