"""The Gaussian sweep's acceptance as one comparison, rz(x) < 2^(32 + y) with y =
-2 beta log2(e) s h: for y >= 0 (Delta E <= 0) every draw passes, because the
device's exponential of every fp32 argument from 32 up is at least 2^32, and
rz(x) of a 32-bit x at most 2^32 - 256.  All 1.04e9 arguments, infinity among
them (a child program with the kernels' own function)."""
import os
import subprocess

import pytest

from paper_1501_05630_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include "icm_internal.h"
#include "icm_device.cuh"
#include <cstdio>
__global__ void check(uint32_t first, uint32_t n, unsigned long long *below)
{
    for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        if (!(icm::ex2_approx(__uint_as_float(first + i)) >= 4294967296.f)) atomicAdd(below, 1ull);
}
int main()
{
    unsigned long long *d, below = 1;
    const uint32_t first = 0x42000000u, last = 0x7f800000u;   // 32 and infinity
    if (cudaMalloc(&d, 8) || cudaMemset(d, 0, 8)) return 2;
    check<<<1216, 256>>>(first, last - first + 1, d);
    if (cudaMemcpy(&below, d, 8, cudaMemcpyDeviceToHost)) return 3;
    printf("%llu\n", below);
    return 0;
}
"""


def test_every_downhill_draw_passes(tmp_path):
    (tmp_path / "t.cu").write_text(SRC)
    subprocess.run([B._nvcc(), *B.ARCH, "-std=c++17", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"),
                    str(tmp_path / "t.cu"), "-o", str(tmp_path / "t")], check=True)
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and int(r.stdout) == 0, r.stdout
