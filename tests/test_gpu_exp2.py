"""The attention kernels' 2^x on the FMA pipe (ex2_pair_fma) by itself, against numpy in 64 bits."""
import ctypes as C
import subprocess

import numpy as np
import pytest
import torch

from paper_2603_08899_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
__global__ void kernel(const float* x, float* y, int pairs)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= pairs) return;
    float a = x[2 * i], b = x[2 * i + 1];
    confu::ex2_pair_fma(a, b);
    y[2 * i] = a;
    y[2 * i + 1] = b;
}
extern "C" int run(const float* x, float* y, int pairs, void* stream)
{
    kernel<<<(pairs + 255) / 256, 256, 0, (cudaStream_t)stream>>>(x, y, pairs);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def exp2_pair(tmp_path_factory):
    d = tmp_path_factory.mktemp("exp2")
    (d / "exp2.cu").write_text(SOURCE)
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", "-cudart", "static", "-o", str(d / "exp2.so"), str(d / "exp2.cu")],
                   check=True)
    L = C.CDLL(str(d / "exp2.so"))

    def run(x):
        assert x.dtype == np.float32 and x.size % 2 == 0
        dx = torch.from_numpy(x).cuda()
        dy = torch.empty_like(dx)
        rc = L.run(C.c_void_p(dx.data_ptr()), C.c_void_p(dy.data_ptr()), C.c_int(x.size // 2), C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        return dy.cpu().numpy()
    return run


def test_error_bound_over_the_arguments_of_weights(exp2_pair):
    # The polynomial is within 2.2e-7 of 2^f; the multiplication by 2^n is exact down to 2^-126 and rounds to a multiple of 2^-149
    # (2^-23 of 2^-126) below.
    x = np.linspace(-126.49, 8.0, 2_000_000, dtype=np.float32)
    want = np.exp2(x.astype(np.float64))
    err = np.abs(exp2_pair(x).astype(np.float64) - want) / np.maximum(want, 2.0 ** -126)
    assert err.max() <= 2.2e-7


def test_exact_at_whole_numbers_and_zero_below(exp2_pair):
    n = np.arange(-126, 8, dtype=np.float32)
    assert np.all(np.abs(exp2_pair(n) / np.exp2(n) - 1) <= 2.0 ** -23)
    x = np.array([-126.51, -127, -127.3, -130, -500, -3e38, -np.inf, -np.inf], dtype=np.float32)
    assert np.all(exp2_pair(x).view(np.uint32) == 0)


def test_nan_stays_nan(exp2_pair):
    x = np.array([np.nan, -3.0, 1.5, np.nan, np.nan, -np.inf, -np.inf, np.nan], dtype=np.float32)
    assert np.array_equal(np.isnan(exp2_pair(x)), np.isnan(x))
