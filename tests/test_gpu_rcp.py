"""The backward walk's reciprocal is the correctly rounded one, for every binary32 value of its
range (a pixel's transmittance before an entry is T / (1 - alpha), 1 - alpha in [0.00999, 1])."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include "fgs_internal.cuh"
#include <cstdio>
__global__ void compare(uint32_t lo, uint32_t hi, unsigned long long* out)
{
    unsigned long long n = 0, differ = 0;
    for (uint32_t b = lo + blockIdx.x * blockDim.x + threadIdx.x; b <= hi; b += gridDim.x * blockDim.x, ++n)
        differ += __float_as_uint(fgs::rcp1(__uint_as_float(b))) != __float_as_uint(__frcp_rn(__uint_as_float(b)));
    atomicAdd(out, n);
    atomicAdd(out + 1, differ);
}
int main()
{
    unsigned long long *d, h[2] = {0, 0};
    if (cudaMalloc(&d, sizeof h) != cudaSuccess || cudaMemset(d, 0, sizeof h) != cudaSuccess) return 1;
    compare<<<608, 256>>>(0x3C000000u, 0x3F800000u, d);            // 1/128 to 1
    if (cudaMemcpy(h, d, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    std::printf("%llu %llu", h[0], h[1]);
}
"""


def test_every_value(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_23891_gb300 import build
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    (tmp_path / "rcp.cu").write_text(SOURCE)
    exe = str(tmp_path / "rcp")
    subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, str(tmp_path / "rcp.cu"), "-o", exe], check=True)
    n, differ = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert n == 0x3F800000 - 0x3C000000 + 1 and differ == 0
