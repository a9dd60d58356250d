"""Device arithmetic of pt_math.h against CUDA's own, on the GPU: small programs
compiled from the header.  The reciprocal over every significand; the transition
matrices from FP32 pairs against the FP64 sums they stand for."""
from __future__ import annotations

import subprocess

import numpy as np
import pytest

from paper_1811_11007_gb300 import build, pt

pytestmark = pytest.mark.gpu

RCP = r"""
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
    unsigned long long* p;
    cudaMallocManaged(&p, 8);
    *p = 0;
    rcp<<<608, 256>>>(p);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    printf("%llu\n", *p);
}
"""

# models as data: lam [4], W [16][4], per model; t from 2^-14 to 2^7 (t |lam| >= 3e-5 as the solver asks)
PMAT = r"""
#include <cstdio>
#include "pt_math.h"
__constant__ double LAM[%(n)d][4] = {%(lam)s};
__constant__ double WW[%(n)d][64] = {%(W)s};
__global__ void pm(unsigned long long* out) {
    __shared__ pt::Exp2Tab tab;
    tab.init();
    __syncthreads();
    const int N = 1 << 21;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
        for (int m = 0; m < %(n)d; ++m) {
            const pt::F2 t = pt::f2_of(exp2(-14.0 + 21.0 * (i + 0.37) / N));
            const double td = (double)t.h + (double)t.l;
            pt::F2 em[4];
            double ex[4] = {1.0, 0, 0, 0};
            bool small = false;
            for (int k = 1; k < 4; ++k) {
                const pt::F2 x = pt::f2_mul(pt::f2_of(LAM[m][k]), t);
                em[k] = x.h > -80.f ? pt::expm1_pair(x, tab) : pt::F2{-1.f, 0.f};
                ex[k] = exp(LAM[m][k] * td);
                small = small || t.h * (float)fabs(LAM[m][k]) <= 3e-5f;
            }
            if (small) continue;
            for (int ij = 0; ij < 16; ++ij) {
                pt::F2 w[4];
                double acc = WW[m][ij * 4];
                for (int k = 1; k < 4; ++k) {
                    w[k] = pt::f2_of(WW[m][ij * 4 + k]);
                    acc = fma(WW[m][ij * 4 + k], ex[k], acc);
                }
                bool sure;
                const float v = pt::p_entry_pair(ij %% 5 == 0 ? 1.f : 0.f, w, em, 1, sure);
                atomicAdd(&out[0], 1ull);
                if (!sure) atomicAdd(&out[1], 1ull);
                else if (v != (float)acc) atomicAdd(&out[2], 1ull);
            }
        }
}
int main() {
    unsigned long long* p;
    cudaMallocManaged(&p, 24);
    p[0] = p[1] = p[2] = 0;
    pm<<<608, 128>>>(p);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    printf("%%llu %%llu %%llu\n", p[0], p[1], p[2]);
}
"""


def _run(tmp_path, text):
    src, exe = tmp_path / "m.cu", tmp_path / "m"
    src.write_text(text)
    subprocess.run([build.NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    return [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]


def test_reciprocal(tmp_path):
    assert _run(tmp_path, RCP) == [0]  # the same bits as __frcp_rn


def test_pair_matrices_round_as_fp64(tmp_path):
    rng = np.random.default_rng(5)
    lam, W = [], []
    for k in range(6):
        exch = np.ones(6) if k == 0 else rng.dirichlet(np.ones(6))
        pi = np.full(4, 0.25) if k == 0 else rng.dirichlet(np.full(4, 5.0))
        l, R = pt.model_eigen(exch, pi)
        for rate in (0.0334, 1.0, 2.9):  # category rates at shape 0.5
            lam.append(l * rate)
            W.append(np.einsum("i,j,ik,jk->ijk", 1 / np.sqrt(pi), np.sqrt(pi), R, R).reshape(64))
    rows = lambda a: ", ".join("{" + ", ".join(float(x).hex() for x in r) + "}" for r in a)  # noqa: E731
    total, unsure, wrong = _run(tmp_path, PMAT % {"n": len(lam), "lam": rows(lam), "W": rows(W)})
    assert total > 10 ** 8
    assert wrong == 0        # a rounding that passes the test is the FP64 sum's
    assert unsure < total // 200
