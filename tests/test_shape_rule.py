"""The rule for launch shapes (shape_lanes in pt_internal.h, compiled for the host) over
every CTA size that a configuration accepts: whole warps, whole virtual threads in a warp,
and each site of an item with exactly one lane."""
from __future__ import annotations

import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_1811_11007_gb300 import build

SRC = r"""
#include "pt_internal.h"
extern "C" int lanes(int vt, int vk, int kp, int pt, int J) { return pt::shape_lanes(vt, vk, kp, pt, J); }
extern "C" int share(int P, int vk) { return pt::cluster_sites(P, vk); }
extern "C" int local(int P, int vt, int vk, int lanes, int pt) { return pt::geo_local(P, pt::Geo{vt, vk, lanes}, pt); }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "r.cpp").write_text(SRC)
    subprocess.run([build.NVCC, "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, str(d / "r.cpp"),
                    "-o", str(d / "r.so")], check=True)
    return C.CDLL(str(d / "r.so"))


@pytest.mark.parametrize("vt", range(32, 513, 32))
def test_shapes_are_whole_warps_and_cover_every_site(rule, vt):
    offered = 0
    for vk in (1, 2, 4, 8):
        for P in (1, vt - 1, vt + 1, 816, 5908):
            Ps = rule.share(P, vk)
            J = -(-Ps // vt)
            for kp in (1, 2, 4, 8):
                for pt in (vt, vt // 2):
                    n = rule.lanes(vt, vk, kp, pt, J)
                    if n == 0:
                        continue
                    offered += 1
                    assert pt % 32 == 0 and 32 % n == 0 and kp * pt == vk * vt * n
                    # the sites of each lane, and where its CTA keeps them
                    cap, seen = rule.local(P, vt, vk, n, pt), np.zeros(P, int)
                    for r in range(kp):
                        t = np.arange(pt)
                        gv = (r * pt + t) // n
                        start = np.minimum(P, gv // vt * Ps)
                        size = np.minimum(P, start + Ps) - start
                        for m in range(-(-Ps // (vt * n))):
                            i = gv % vt + vt * (t % n) + m * vt * n
                            on = i < size
                            seen[(start + i)[on]] += 1
                            assert not on.any() or (t + m * pt)[on].max() < cap
                    assert (seen == 1).all()
    assert offered
