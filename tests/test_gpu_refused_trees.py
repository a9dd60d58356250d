"""Edge lists whose degrees are a tree's but which are none: only the device sees it, after
kernels that follow the canonical arrays have been queued."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu
N = 6
BAD = np.array([(0, 6), (1, 6), (2, 6), (3, 7), (4, 8), (5, 9), (7, 8), (8, 9), (9, 7)], np.int32)


def _setup():
    a = synth.simulate(N, 200, 53, model="gtr", alpha=0.5, mean_branch=0.1)
    ctx = pt.Context(precision="mixed", table_log2=12)
    aid = ctx.load_alignment(a.codes)
    ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
    return ctx, aid, np.stack([a.tree_edges, BAD]).astype(np.int32), np.full((2, 2 * N - 3), 0.1)


def _reach(e, l):
    """The keys of a tree and of its neighbours."""
    return {oracle.tree_key(N, e)} | {oracle.tree_key(N, x) for x in oracle.nni_neighbours(N, e, l)[0]}


def test_a_recorded_round_refuses_them():
    ctx, aid, e, l = _setup()
    with ctx:
        g = ctx.graph([aid], [4], [10.0])
        try:
            with pytest.raises(pt.PTError) as ex:
                g.run([g.set_frontier(0, e, l)], [-1e300])
            assert ex.value.status == 1
            seen = {tuple(int(x) for x in k) for k in ctx.visited(aid)["keys"]}
            assert seen <= _reach(e[0], l[0])  # nothing of the refused one entered the table
            ctx.reset_visited(aid)  # and the round works on the good one
            lm, _ = g.run([g.set_frontier(0, e[:1], l[:1])], [-1e300])
            got = {k: np.array(v) for k, v in g.next(0).items()}
        finally:
            g.close()
        ctx.reset_visited(aid)
        lm2, want = ctx.expand(aid, e[:1], l[:1], 10.0, -1e300)
    assert lm[0] == lm2 and len(want["keys"])
    for k in want:
        np.testing.assert_array_equal(got[k], want[k])


def test_a_round_refuses_them():
    ctx, aid, e, l = _setup()
    with ctx:
        ctx.begin(aid, e[:1], l[:1], 10.0)
        with pytest.raises(pt.PTError) as ex:
            ctx.expand(aid, e, l, 10.0, -1e300)
        assert ex.value.status == 1
        seen = {tuple(int(x) for x in k) for k in ctx.visited(aid)["keys"]}
        assert seen <= _reach(e[0], l[0])
