"""The Newton exchange of a cluster's CTA on the host (exchange_warps.cpp compiles the kernel's
own code): whichever warp runs ahead, and also after a wait has run out, every warp sees the
same number of evaluations and no barrier is left waiting."""
from __future__ import annotations

import ctypes as C
import itertools
import os
import subprocess

import numpy as np
import pytest

from paper_1811_11007_gb300 import build


@pytest.fixture(scope="module")
def exchange(tmp_path_factory):
    so = tmp_path_factory.mktemp("exchange") / "exchange.so"
    src = os.path.join(os.path.dirname(__file__), "exchange_warps.cpp")
    subprocess.run([build.NVCC, "-std=c++17", "-O1", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, src, "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))

    def run(nw, ld, turn, solves, steps, maxit, drop, starve=0):
        evals, up = np.full((solves, 32 * nw), -1, np.int32), C.c_int(-1)
        t = np.array(turn, np.int32)
        rc = L.exchange_warps(nw, ld, t.ctypes.data_as(C.c_void_p), solves, steps, maxit, drop, starve,
                              evals.ctypes.data_as(C.c_void_p), C.byref(up))
        assert rc == 0, {1: "no thread can go on", 2: "too many arrivals at a barrier"}[rc]
        assert (evals == evals[:, :1]).all(), "warps disagree on the evaluations of a solve"
        return evals[:, 0].tolist(), up.value
    return run


def _orders(nw):
    return itertools.permutations(range(nw)) if nw <= 3 else [range(nw), range(nw - 1, -1, -1), [1, 0, *range(2, nw)]]


@pytest.mark.parametrize("nw", [1, 2, 3, 8])
@pytest.mark.parametrize("steps,maxit", [(3, 50), (1, 50), (9, 4)])
def test_every_order_takes_the_same_evaluations(exchange, nw, steps, maxit):
    for ld in range(min(nw, 4)):
        for turn in _orders(nw):
            assert exchange(nw, ld, turn, 5, steps, maxit, 1000) == ([min(steps, maxit)] * 5, 0)


@pytest.mark.parametrize("nw", [1, 2, 3, 8])
@pytest.mark.parametrize("drop", [0, 1, 2, 3, 7])
def test_a_wait_that_runs_out_ends_the_solve_for_every_warp(exchange, nw, drop):
    """Three evaluations a solve; the sums of exchange `drop` and of later ones never arrive: the solve
    ends with that evaluation, and no later one is made."""
    want = [3 if s < drop // 3 else drop % 3 + 1 if s == drop // 3 else 0 for s in range(5)]
    for ld in range(min(nw, 4)):
        for turn in _orders(nw):
            assert exchange(nw, ld, turn, 5, 3, 50, drop) == (want, 1)


@pytest.mark.parametrize("nw", [2, 3, 8])
def test_a_warp_slower_than_the_wait(exchange, nw):
    """The leader gives up on its own CTA's last warp, which then finds the same end."""
    for ld in range(min(nw, 4)):
        for turn in _orders(nw):
            if turn[-1] != ld:
                assert exchange(nw, ld, turn, 5, 3, 50, 1000, starve=1) == ([1, 0, 0, 0, 0], 1)
