"""The field sum behind the mean of every correction (k_sum in sums.cuh), compiled by itself: FP32 data is
added four additions deep and in FP64 beyond that.

Tolerance: four roundings of 2^-24 of a sum of positive values, 2^-22 of it, whatever the length; a running
FP32 sum per thread is off by up to 2^-25 of itself per addition, which equal values add up (values on
which it fails the bound are among these).
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "sums.cuh"
using namespace pmeft;
template <typename T>
static int run(const T* x, long long total, int grid, double* out)
{
    double *part = nullptr, *fin = nullptr;
    cudaMalloc(&part, sizeof(double) * kPartialsDoubles);
    cudaMalloc(&fin, sizeof(double) * 16);
    cudaMemset(part, 0, sizeof(double) * kPartialsDoubles);
    k_sum<T><<<grid, 256>>>(x, (size_t)total, part, fin);
    const cudaError_t e = cudaMemcpy(out, fin, sizeof(double) * 2, cudaMemcpyDeviceToHost);
    cudaFree(part);
    cudaFree(fin);
    return (int)e;
}
extern "C" int sum32(const float* x, long long t, int g, double* o) { return run(x, t, g, o); }
extern "C" int sum64(const double* x, long long t, int g, double* o) { return run(x, t, g, o); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("sums")
    (d / "s.cu").write_text(SRC)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                    "--expt-relaxed-constexpr", "-shared", "-I", ROOT + "/include", "-I",
                    ROOT + "/paper_2604_15434_gb300/csrc", "-o", str(d / "s.so"), str(d / "s.cu")], check=True)
    return ctypes.CDLL(str(d / "s.so"))


def total(lib, x, grid):
    out = (ctypes.c_double * 2)()
    fn = lib.sum32 if x.dtype == torch.float32 else lib.sum64
    torch.cuda.synchronize()
    assert fn(ctypes.c_void_p(x.data_ptr()), ctypes.c_longlong(x.numel()), grid, out) == 0
    return out[0], out[1]


@pytest.mark.parametrize("n,grid", [(8, 2), (64, 608), (512, 608), (512, 32)])
@pytest.mark.parametrize("kind", ["equal", "random"])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_sum(lib, n, grid, kind, dtype):
    rng = np.random.default_rng(n + grid)
    for v in rng.uniform(1.0, 2.0, 4):
        if kind == "equal":
            x = torch.full((n ** 3,), v, dtype=dtype, device="cuda")
        else:
            x = (torch.rand(n ** 3, dtype=torch.float64, device="cuda") + v).to(dtype)
        want = float(x.double().sum())
        got, mean = total(lib, x, grid)
        assert abs(got - want) <= (2.0 ** -22 if dtype == torch.float32 else 1e-13) * want
        assert abs(mean * n ** 3 - got) <= 1e-15 * got
