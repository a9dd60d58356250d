"""Contexts of several host threads at once: each launch asks for its own amount of shared
memory, whatever another thread's launch of the same kernel asks for meanwhile."""
from __future__ import annotations

import threading

import numpy as np
import pytest

from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu


def _ctx(n, sites):
    a = synth.simulate(n, sites, 71 + n, model="gtr", alpha=0.5, mean_branch=0.05)
    ctx = pt.Context(precision="mixed", table_log2=14, full_max_sweeps=1)
    aid = ctx.load_alignment(a.codes)
    ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
    return ctx, aid, a.tree_edges[None], np.full((1, 2 * n - 3), 0.05)


# lengths given: matrices of all edges in shared memory; optimised: the sum-table too; proposals
# (a neighbourhood that keeps nothing): partials and the proposal kernel
@pytest.mark.parametrize("what,times", [("fixed", 1500), ("full", 150), ("expand", 60)])
def test_contexts_of_two_threads(what, times):
    made = [_ctx(6, 60), _ctx(90, 1500)]
    bad = []

    def call(ctx, aid, e, l):
        if what != "expand":
            return ctx.score(aid, e, l, what)[0][0]
        ctx.reset_visited(aid)
        ctx.expand(aid, e, l, 0.0, 0.0)
        return float(np.sort(ctx.last_proposals()["lnl"])[-1])

    def work(k, want):
        try:
            for _ in range(times):
                got = call(*made[k])
                if got != want:
                    bad.append((k, got, want))
        except Exception as x:  # noqa: BLE001
            bad.append((k, repr(x)))
    try:
        want = [call(*m) for m in made]
        ts = [threading.Thread(target=work, args=(k, want[k])) for k in range(2)]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
    finally:
        for m in made:
            m[0].close()
    assert not bad, bad[:3]
