"""The factors that join the parts of a row's sums in the acceptance walks (joint, joint_f32), against numpy in extended precision."""
import ctypes as C
import subprocess

import numpy as np
import pytest
import torch

from paper_2603_08899_b200 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "walk.cuh"
__global__ void kernel(const float* d, float k, double* y64, float* y32, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y64[i] = confu::walk::joint(d[i], (double)k);
    y32[i] = confu::walk::joint_f32(d[i], k);
}
extern "C" int run(const float* d, float k, double* y64, float* y32, int n, void* stream)
{
    kernel<<<(n + 255) / 256, 256, 0, (cudaStream_t)stream>>>(d, k, y64, y32, n);
    return (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def factors(tmp_path_factory):
    d = tmp_path_factory.mktemp("joint")
    (d / "joint.cu").write_text(SOURCE)
    subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-shared", "-cudart", "static", "-o", str(d / "joint.so"), str(d / "joint.cu")],
                   check=True)
    L = C.CDLL(str(d / "joint.so"))

    def run(x, k):
        dx = torch.from_numpy(x).cuda()
        y64, y32 = torch.empty(x.size, dtype=torch.float64, device="cuda"), torch.empty(x.size, device="cuda")
        rc = L.run(C.c_void_p(dx.data_ptr()), C.c_float(k), C.c_void_p(y64.data_ptr()), C.c_void_p(y32.data_ptr()), C.c_int(x.size),
                   C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert rc == 0
        return y64.cpu().numpy(), y32.cpu().numpy()
    return run


@pytest.mark.parametrize("temperature", [1.0, 0.7, 0.05])
def test_error_bounds(factors, temperature):
    k = np.float32(np.float32(1.0 / temperature) * np.float32(1.4426950408889634))
    x = np.concatenate([-np.logspace(-6, 2, 300_001), -np.linspace(0, 40, 300_001)]).astype(np.float32)
    arg = x.astype(np.longdouble) * np.longdouble(k)
    whole = np.rint(arg)
    want = np.exp((arg - whole) * np.log(np.longdouble(2)))
    y64, y32 = factors(x, k)
    keep = arg > -120
    # power series: 7e-12; rounding of fp64 sums and of the product d k: 2^-53 times 1 + |d k|, times ln 2
    assert np.abs(np.ldexp(y64[keep].astype(np.longdouble), -whole[keep].astype(int)) / want[keep] - 1).max() <= 1e-11
    # half a unit for the last sum, the rest for the roundings in front of it: 1.3 * 2^-24 at most
    assert np.abs(np.ldexp(y32[keep].astype(np.longdouble), -whole[keep].astype(int)) / want[keep] - 1).max() <= 1.3 * 2.0 ** -24


def test_ends(factors):
    y64, y32 = factors(np.array([0.0, -np.inf, -1e30, -3e38], dtype=np.float32), np.float32(1.4426950408889634))
    assert y64.tolist() == [1, 0, 0, 0] and y32.tolist() == [1, 0, 0, 0]
