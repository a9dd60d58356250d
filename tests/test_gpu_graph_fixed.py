"""Recorded rounds whose visits take no sweep."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu


def _round(sweeps):
    n = 12
    a = synth.simulate(n, 500, 47, model="gtr", alpha=0.5, mean_branch=0.1)
    with pt.Context(precision="mixed", table_log2=14, full_max_sweeps=sweeps) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
        lmax, f = ctx.begin(aid, a.tree_edges[None], np.full((1, 2 * n - 3), 0.1), 30.0)
        g = ctx.graph([aid], [8], [30.0])
        try:
            nf = g.set_frontier(0, f["edges"], f["lengths"])
            lm, _ = g.run([nf], [lmax])
            launches = ctx.stats()["launches"]
            got = {k: np.array(v) for k, v in g.next(0).items()}
        finally:
            g.close()
        ctx.reset_visited(aid)
        lm2, want = ctx.expand(aid, f["edges"], f["lengths"], 30.0, lmax)
    assert lm[0] == lm2 and len(want["keys"]) > 0
    for k in want:
        np.testing.assert_array_equal(got[k], want[k])
    return launches


def test_visits_without_sweeps_are_only_scored():
    """In mixed precision such a visit is its score: no optimisation kernel is recorded."""
    assert _round(0) < _round(1)
