"""The kernels' reciprocal of a row's sum against the division, over all mantissas."""
import ctypes
import os
import subprocess

import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "das_tc.h"
__global__ void kernel(const float *x, float *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = das::tc::inverse(x[i]);
}
extern "C" int run(const float *x, float *y, int n) {
    kernel<<<(n + 255) / 256, 256>>>(x, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("inverse")
    (d / "inverse.cu").write_text(SOURCE)
    from paper_2609_34538_gb300 import build
    subprocess.run([build.NVCC, *build.ARCH, *build.FLAGS, "-shared", str(d / "inverse.cu"), "-o",
                    str(d / "inverse.so")], check=True, capture_output=True)
    return ctypes.CDLL(str(d / "inverse.so"))


def run(lib, x):
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    assert lib.run(ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()), x.numel()) == 0
    return y


@pytest.mark.parametrize("exponent", [0, 1, 20, 119])
def test_within_an_ulp_of_the_division(lib, exponent):
    bits = torch.arange(1 << 23, dtype=torch.int32, device="cuda") + ((127 + exponent) << 23)
    x = bits.view(torch.float32)
    ulps = (run(lib, x).view(torch.int32) - (1.0 / x).view(torch.int32)).abs()
    assert int(ulps.max()) <= 1


def test_no_sum(lib):
    x = torch.tensor([0.0, float("nan")], device="cuda")
    assert run(lib, x).tolist() == [0.0, 0.0]
