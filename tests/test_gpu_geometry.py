"""Summation geometries other than the default's: CTA sizes whose warps are no power of two
or that cannot be halved, and large problems whose sites are split into shares.  A tree's or
a neighbour's result is the same, bit for bit, whatever shape the number of items picks."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu


def _case(n, sites, trees, branch):
    a = synth.simulate(n, sites, 177 + n, model="gtr", alpha=0.5, mean_branch=branch)
    rng = np.random.default_rng(n)
    e = np.stack([synth.reinsert_leaves(a.tree_edges, n, 2, rng) for _ in range(trees)])
    return a, np.ascontiguousarray(e, np.int32), rng.exponential(branch, (trees, 2 * n - 3)) + 1e-3


def _props(ctx, aid, e, l):
    ctx.reset_visited(aid)
    ctx.expand(aid, e, l, 0.0, 0.0)  # keeps nothing: proposals only
    p = ctx.last_proposals()
    return {(int(p["parent"][i]),) + tuple(int(x) for x in p["keys"][i]): (p["lnl"][i], *p["len5"][i])
            for i in range(len(p["lnl"]))}


def _check(ctx, aid, e, l, counts):
    lnl, lens, _ = ctx.score(aid, e, l, "full")
    many = _props(ctx, aid, e[:40], l[:40])
    for k in counts:
        lnl_k, lens_k, _ = ctx.score(aid, e[:k], l[:k], "full")
        np.testing.assert_array_equal(lnl_k, lnl[:k])
        np.testing.assert_array_equal(lens_k, lens[:k])
        if k >= 40:
            continue
        few = _props(ctx, aid, e[:k], l[:k])
        both = set(few) & set(many)
        assert len(both) >= len(few) // 2  # the others have another proposer in the larger round
        assert all(few[x] == many[x] for x in both)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("threads", [32, 64, 96, 192, 288, 384, 416, 512])
def test_results_do_not_depend_on_the_shape(prec, threads):
    n = 14
    a, e, l = _case(n, 2400, 160, 0.2)
    with pt.Context(precision=prec, table_log2=16, threads=threads, full_max_sweeps=2) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
        assert ctx.alignment_info(aid)[1] > 1024
        _check(ctx, aid, e, l, (1, 2, 5, 19, 75))


# more patterns than one CTA's shared memory holds: shares of the sites in mixed precision,
# a cluster or one CTA with its table in global memory in FP64
@pytest.mark.parametrize("prec,threads", [("mixed", 0), ("mixed", 96), ("mixed", 512), ("fp64", 0)])
def test_large_problems_do_not_depend_on_the_shape(prec, threads):
    n = 16
    a, e, l = _case(n, 8000, 60, 0.25)
    with pt.Context(precision=prec, table_log2=16, threads=threads, full_max_sweeps=1, prop_max_sweeps=2) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
        assert ctx.alignment_info(aid)[1] > 3500  # 68 bytes a pattern in FP32
        _check(ctx, aid, e, l, (1, 4, 19))


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_a_recorded_round_is_the_same_at_every_count(prec):
    """A recorded round issues one launch per shape and the counts decide which one runs: frontiers
    from one tree (every CTA on few items) to more neighbours than the GPU holds at once."""
    n, most = 14, 40
    a, e, l = _case(n, 900, most, 0.1)
    with pt.Context(precision=prec, table_log2=16, full_max_sweeps=2, prop_max_sweeps=2) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, 4)
        g = ctx.graph([aid], [most], [np.inf])  # every neighbour is kept and visited
        try:
            for k in (1, 2, 3, 5, 8, 13, 22, most):
                ctx.reset_visited(aid)
                lm, _ = g.run([g.set_frontier(0, e[:k], l[:k])], [-1e300])
                got = {x: np.array(v) for x, v in g.next(0).items()}
                ctx.reset_visited(aid)
                lm2, want = ctx.expand(aid, e[:k], l[:k], np.inf, -1e300)
                assert lm[0] == lm2 and len(want["keys"]) >= k
                for x in want:
                    np.testing.assert_array_equal(got[x], want[x])
        finally:
            g.close()
