"""The detector's square root against the correctly rounded one, for 0 and every
FP32 value from 1 to 2^64 (the whole range of its arguments)."""

import os
import subprocess

import pytest

from paper_2607_01757_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include "vt_sqrt.cuh"

// bit patterns first .. last; the argument 0 besides
__global__ void check(unsigned first, unsigned last, unsigned long long *wrong, unsigned long long *seen) {
    unsigned long long w = 0, n = 0;
    for (unsigned long long b = first + blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; b <= last;
         b += (unsigned long long)gridDim.x * blockDim.x) {
        const float q = __uint_as_float((unsigned)b);
        w += __float_as_uint(vt::sqrt_score(q)) != __float_as_uint(__fsqrt_rn(q));
        ++n;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) w += __float_as_uint(vt::sqrt_score(0.0f)) != 0u;
    atomicAdd(wrong, w);
    atomicAdd(seen, n);
}

int main() {
    unsigned long long *c, h[2] = {1, 0};
    if (cudaMallocManaged(&c, 16) != cudaSuccess) return 2;
    c[0] = c[1] = 0;
    check<<<1216, 256>>>(0x3f800000u, 0x5f800000u, c, c + 1);  // 1 .. 2^64
    if (cudaDeviceSynchronize() != cudaSuccess) return 3;
    h[0] = c[0], h[1] = c[1];
    printf("%llu %llu\n", h[0], h[1]);
    return 0;
}
"""


def test_every_argument(tmp_path):
    src, exe = tmp_path / "sqrt.cu", str(tmp_path / "sqrt")
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, "-O3", "-std=c++17", "-I", build.CSRC, str(src), "-o", exe], check=True,
                   timeout=300)
    assert os.path.exists(exe)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout.split()
    assert out == ["0", str(64 * 2**23 + 1)], out
