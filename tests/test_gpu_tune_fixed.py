"""Scores at given lengths run no Newton solve, so they have nothing to tune."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_fixed_scores_leave_the_bucket_untuned(prec, tmp_path):
    n, trees = 10, 400  # more than two trees per SM: enough to tune on
    a = synth.simulate(n, 300, 43, model="gtr", alpha=0.5, mean_branch=0.1)
    e, l = synth.random_trees(n, trees, 5)
    with pt.Context(precision=prec, table_log2=12, full_max_sweeps=1) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
        ctx.autotune(True, str(tmp_path / "tune.json"))
        fixed = ctx.score(aid, e, l, "fixed")[0]
        assert not any(v["full_threads"] for v in ctx.autotune_report().values())
        ctx.score(aid, e, l, "full")
        (v,) = ctx.autotune_report().values()
        assert v["full_threads"] and v["full_items"] == trees
        if prec == "mixed":  # summed in units of their own; FP64 sums in the tuned geometry
            np.testing.assert_array_equal(ctx.score(aid, e, l, "fixed")[0], fixed)
