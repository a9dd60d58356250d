"""The canonicaliser's warp on the host (canon_lanes.cpp compiles the kernel's own code):
the canonical form must not depend on the order in which the lanes run between two of
the warp's barriers."""
from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_1811_11007_gb300 import build, synth

UPD = 1 << 16  # schedule entry: refresh instead of visit


@pytest.fixture(scope="module")
def canon(tmp_path_factory):
    so = tmp_path_factory.mktemp("canon") / "canon.so"
    src = os.path.join(os.path.dirname(__file__), "canon_lanes.cpp")
    subprocess.run([build.NVCC, "-std=c++17", "-O1", "-shared", "-Xcompiler", "-fPIC", "-I", build.CSRC, src, "-o",
                    str(so)], check=True)
    L = C.CDLL(str(so))

    def run(n, edges, lengths, order):
        NN, E = 2 * n - 2, 2 * n - 3
        e, l = np.ascontiguousarray(edges, np.int32), np.ascontiguousarray(lengths, np.float64)
        out = {"up": np.full(NN, -7, np.int32), "ch": np.full((NN, 2), -7, np.int32), "len": np.full(NN, -7.0),
               "bits": np.full((NN, 2), 7, np.uint64), "erank": np.full(NN, -7, np.int32),
               "sched": np.full(3 * n, -7, np.int32), "key": np.full(2, 7, np.uint64), "emap": np.full(E, -7, np.int32),
               "err": np.zeros(8, np.int32)}
        p = [x.ctypes.data_as(C.c_void_p) for x in (e, l)] + [C.c_uint(order)] + \
            [x.ctypes.data_as(C.c_void_p) for x in out.values()]
        assert L.canon_lanes(C.c_int(n), *p) == 0, "lanes met at different warp-wide calls"
        return out
    return run


def _expect(n, edges, lengths):
    """The canonical form by recursion."""
    adj = {}
    for k, (a, b) in enumerate(np.asarray(edges).tolist()):
        adj.setdefault(a, []).append((b, k))
        adj.setdefault(b, []).append((a, k))
    NN, E = 2 * n - 2, 2 * n - 3
    f = {"up": np.full(NN, -1, np.int32), "ch": np.full((NN, 2), -1, np.int32), "len": np.zeros(NN),
         "bits": np.zeros((NN, 2), np.uint64), "erank": np.full(NN, -1, np.int32), "emap": np.zeros(E, np.int32)}
    sched, sets, fresh = [], {}, iter(range(n, NN))

    def leaves(v, p):
        if v < n:
            return frozenset([v])
        return frozenset().union(*(leaves(c, v) for c, _ in adj[v] if c != p))

    def walk(v, p, pc, k):
        c = v if v < n else next(fresh)
        below = leaves(v, p)
        f["up"][c], f["len"][c], f["emap"][k] = pc, lengths[k], c
        for t in below:
            f["bits"][c, t // 64] |= np.uint64(1 << (t % 64))
        sched.append(c)
        if v >= n:
            kids = sorted(((x, j) for x, j in adj[v] if x != p), key=lambda x: min(leaves(x[0], v)))
            f["ch"][c] = [walk(x, v, c, j) for x, j in kids]
            if p != 0:
                sets[c] = sum(1 << t for t in below)
            sched.append(c | UPD)
        return c
    (top, k0), = adj[0]
    f["bits"][0, 0] = 1
    walk(top, 0, 0, k0)
    for r, c in enumerate(sorted(sets, key=sets.get)):
        f["erank"][c] = r
    f["sched"] = np.array(sched + [-1] * (3 * n - len(sched)), np.int32)
    f["key"] = np.array(oracle.tree_key(n, edges), np.uint64)
    f["err"] = np.zeros(8, np.int32)
    return f


def _caterpillar(n):
    leaf = [(v, n if v == 0 else 2 * n - 3 if v == n - 1 else n + v - 1) for v in range(n)]
    return np.array(leaf + [(n + i, n + i + 1) for i in range(n - 3)], np.int32)


@pytest.mark.parametrize("n", [3, 4, 5, 9, 27, 33, 64, 128])
def test_canonical_form_does_not_depend_on_lane_order(canon, n):
    rng = np.random.default_rng(n)
    trees = [_caterpillar(n)] + [synth.relabel_inner(synth.random_topology(n, rng), n, rng) for _ in range(3)]
    for e in trees:
        l = rng.exponential(0.1, 2 * n - 3)
        want = _expect(n, e, l)
        for order in (0, 1, 2, 3, 4):
            got = canon(n, e, l, order)
            for x in want:
                np.testing.assert_array_equal(got[x], want[x], err_msg="%s, lane order %d" % (x, order))


# edge lists that are no trees; the last three have a tree's degrees
BAD = {
    "self-loop": (5, [(0, 5), (1, 5), (5, 5), (2, 6), (6, 7), (3, 7), (4, 7)]),
    "node out of range": (4, [(0, 4), (1, 4), (4, 5), (2, 5), (3, 6)]),
    "negative node": (4, [(0, 4), (1, 4), (4, 5), (2, 5), (3, -1)]),
    "leaf of degree two": (5, [(0, 5), (1, 5), (5, 6), (2, 6), (6, 7), (3, 7), (3, 4)]),
    "cycle beside leaf 0's part": (6, [(0, 6), (1, 6), (2, 6), (3, 7), (4, 8), (5, 9), (7, 8), (8, 9), (9, 7)]),
    "cycle in leaf 0's part": (6, [(3, 6), (4, 6), (5, 6), (0, 7), (1, 8), (2, 9), (7, 8), (8, 9), (9, 7)]),
    "double edge in leaf 0's part": (5, [(2, 5), (3, 5), (4, 5), (6, 7), (7, 6), (0, 6), (1, 7)]),
}


@pytest.mark.parametrize("what", sorted(BAD))
def test_a_list_that_is_no_tree_leaves_a_tree_behind(canon, what):
    """Flagged, with the key 0, and with arrays that every later kernel can follow: a caterpillar's."""
    n, e = BAD[what]
    want = _expect(n, _caterpillar(n), np.full(2 * n - 3, 0.1))
    want["key"][:] = 0
    want["err"][0] = 1  # tree index + 1
    for order in (0, 1, 2, 3):
        got = canon(n, e, np.full(2 * n - 3, 0.3), order)
        for x in want:
            np.testing.assert_array_equal(got[x], want[x], err_msg=x)
