"""Transition matrices from FP32 pairs under strongly uneven base frequencies: an entry
whose rounding test passes is the FP64 sum's, bit for bit, at the error interval that the
solver gives it."""
from __future__ import annotations

import subprocess

import numpy as np
import pytest

from paper_1811_11007_gb300 import build, pt

pytestmark = pytest.mark.gpu

PMAT = r"""
#include <cstdio>
#include "pt_math.h"
__constant__ double LAM[%(n)d][4] = {%(lam)s};
__constant__ double WW[%(n)d][64] = {%(W)s};
__global__ void pm(unsigned long long* out) {
    __shared__ pt::Exp2Tab tab;
    tab.init();
    __syncthreads();
    const int N = 1 << 20;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x)
        for (int m = 0; m < %(n)d; ++m) {
            const pt::F2 t = pt::f2_of(exp2(-15.0 + 10.0 * (i + 0.37) / N));
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
                const float delta = ij %% 5 == 0 ? 1.f : 0.f;
                bool sure;
                const float v = pt::p_entry_pair(delta, w, em, 1, sure%(base)s);
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
BASE = ", pt::p_entry_base(delta, WW[m] + ij * 4)"


@pytest.mark.parametrize("least", [1e-2, 1e-3, 1e-4])
def test_pair_matrices_round_as_fp64_for_uneven_frequencies(tmp_path, least):
    rng = np.random.default_rng(int(1 / least))
    lam, W = [], []
    for k in range(6):
        exch = rng.dirichlet(np.ones(6))
        pi = rng.dirichlet(np.full(4, 5.0))
        pi[rng.integers(4)] = least
        if k % 2:
            pi[rng.integers(4)] = 3 * least
        pi /= pi.sum()
        l, R = pt.model_eigen(exch, pi)
        for rate in (0.0334, 1.0, 2.9):
            lam.append(l * rate)
            W.append(np.einsum("i,j,ik,jk->ijk", 1 / np.sqrt(pi), np.sqrt(pi), R, R).reshape(64))
    rows = lambda a: ", ".join("{" + ", ".join(float(x).hex() for x in r) + "}" for r in a)  # noqa: E731
    src, exe = tmp_path / "m.cu", tmp_path / "m"
    src.write_text(PMAT % {"n": len(lam), "lam": rows(lam), "W": rows(W), "base": BASE})
    subprocess.run([build.NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True)
    total, unsure, wrong = [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True,
                                                           text=True).stdout.split()]
    assert total > 10 ** 7
    assert wrong == 0
