"""Device arithmetic of pt_math.h against CUDA's own, on the GPU: a small program
compiled from the header runs over every significand."""
from __future__ import annotations

import os
import subprocess

import pytest

from paper_1811_11007_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include "pt_math.h"
// all 2^23 significands at exponents across the range and just outside it, both signs
__global__ void rcp(unsigned long long* bad) {
    const int es[] = {1, 62, 63, 64, 65, 100, 126, 127, 128, 150, 189, 190, 191, 192, 253};
    for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < (1u << 23); m += gridDim.x * blockDim.x)
        for (int e : es)
            for (unsigned s = 0; s < 2; ++s) {
                const float x = __int_as_float((int)((s << 31) | ((unsigned)e << 23) | m));
                if (__float_as_int(pt::rcp_rn(x)) != __float_as_int(__frcp_rn(x))) atomicAdd(bad, 1ull);
            }
}
int main() {
    unsigned long long *p;
    cudaMallocManaged(&p, 8);
    p[0] = 0;
    rcp<<<608, 256>>>(p);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    printf("%llu %llu\n", p[0], p[1]);
}
"""


def test_reciprocal(tmp_path):
    src, exe = tmp_path / "m.cu", tmp_path / "m"
    src.write_text(SRC)
    subprocess.run([build.NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, env=dict(os.environ)).stdout.split()
    assert int(out[0]) == 0  # the same bits as __frcp_rn
