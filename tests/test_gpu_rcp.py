"""The set-up's reciprocal (rcp_newton) against the division, in a kernel of its own."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_10314_gb300", "csrc")
SOURCE = """
#include "smerf_internal.cuh"
__global__ void kernel(const double* x, double* r, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = smerf::rcp_newton(x[i]);
}
extern "C" int run(const double* x, double* r, int n)
{
    kernel<<<(n + 255) / 256, 256>>>(x, r, n);
    return cudaDeviceSynchronize();
}
"""


def test_within_an_ulp_of_the_division(tmp_path):
    """The 20 bits of the approximation become 40 and 80: what is left is the last step's rounding and that
    of its correction, below an ulp together."""
    import torch
    src, lib = str(tmp_path / "rcp.cu"), str(tmp_path / "rcp.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                    "-Xcompiler", "-fPIC", "-I" + CSRC, src, "-o", lib], check=True)
    rng = np.random.default_rng(4)
    m = np.concatenate([rng.uniform(1, 2, 200000), 1 + np.arange(64) * 2.0 ** -52, 2 - np.arange(1, 64) * 2.0 ** -52,
                        np.sqrt(2) * (1 + np.arange(-8, 9) * 2.0 ** -52), 1 + 2.0 ** -np.arange(1, 53)])
    e = rng.integers(-1000, 1001, len(m))
    e[:100000] = rng.integers(-4, 5, 100000)
    x = m * 2.0 ** e * rng.choice([-1.0, 1.0], len(m))
    d = torch.as_tensor(x).cuda()
    r = torch.empty_like(d)
    torch.cuda.synchronize()
    assert ctypes.CDLL(lib).run(ctypes.c_void_p(d.data_ptr()), ctypes.c_void_p(r.data_ptr()), len(x)) == 0
    assert int(np.abs(r.cpu().numpy().view(np.int64) - (1.0 / x).view(np.int64)).max()) <= 1
