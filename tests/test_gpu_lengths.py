"""Starting lengths that FP32 cannot hold: every finite length is accepted, and a solve
that brings one back below tmax counts as a move."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu
N = 10


def _ctx(**kw):
    a = synth.simulate(N, 400, 41, model="gtr", alpha=0.5, mean_branch=0.1)
    ctx = pt.Context(precision="mixed", table_log2=14, **kw)
    aid = ctx.load_alignment(a.codes)
    ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
    return ctx, aid, a.tree_edges[None]


# P(t) is the stationary matrix at all of these and at 1e38, so everything but the length itself is the same
@pytest.mark.parametrize("long", [2.0 ** 128, 1e39, 1e300])
def test_full_optimisation_counts_a_move_from_any_length(long):
    ctx, aid, e = _ctx()
    with ctx:
        _, l, _ = ctx.score(aid, e, np.full((1, 2 * N - 3), 0.1))
        first = int(np.argmax((e[0] == 0).any(1)))  # leaf 0's edge is solved first, and at its optimum nothing else moves

        def run(t):
            x = l.copy()
            x[0, first] = t
            r = ctx.score(aid, e, x)
            return r[0], r[1], ctx.stats()["full_sweeps"]
        want, got = run(1e38), run(long)
        assert want[2] >= 2
        assert got[2] == want[2]
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])


@pytest.mark.parametrize("long", [2.0 ** 128, 1e39, 1e300])
def test_proposals_count_a_move_from_any_length(long):
    ctx, aid, e = _ctx(propose_mode=pt.PROPOSE_CENTRAL)
    with ctx:
        _, l, _ = ctx.score(aid, e, np.full((1, 2 * N - 3), 0.1))
        inner = int(np.argmax((e[0] >= N).all(1)))

        def run(t):
            x = l.copy()
            x[0, inner] = t
            ctx.reset_visited(aid)
            ctx.expand(aid, e, x, 0.0, 0.0)  # keeps nothing: proposals only
            p = ctx.last_proposals()
            return p["lnl"], p["len5"][:, 0], ctx.stats()["prop_sweeps"]
        want, got = run(1e38), run(long)
        assert got[2] == want[2]
        np.testing.assert_array_equal(got[0], want[0])
        np.testing.assert_array_equal(got[1], want[1])
