"""Launch shapes: a tree's or a neighbour's result does not depend on how many
others share the launch, bit for bit (the number of items picks the shape: CTAs
per item and lanes per summing thread)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from paper_1811_11007_gb300 import pt, synth

pytestmark = pytest.mark.gpu


def _case(n, sites, ncat, trees, branch=0.05):
    a = synth.simulate(n, sites, 77 + n, model="gtr", alpha=0.5, mean_branch=branch)
    rng = np.random.default_rng(n)
    e = np.stack([synth.reinsert_leaves(a.tree_edges, n, 2, rng) for _ in range(trees)])
    return a, np.ascontiguousarray(e, np.int32), rng.exponential(branch, (trees, 2 * n - 3)) + 1e-3


# patterns: below one site per thread, at a tile edge and past it, and (24 x 6000 at
# longer branches) more than one CTA's shared memory holds
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,sites,ncat,branch", [(6, 90, 4, 0.1), (12, 600, 1, 0.2), (16, 900, 4, 0.1),
                                                 (24, 6000, 4, 0.15)])
def test_full_optimisation_is_shape_independent(prec, n, sites, ncat, branch):
    a, e, l = _case(n, sites, ncat, 340 if sites < 6000 else 170, branch)
    with pt.Context(precision=prec, table_log2=12, full_max_sweeps=2) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, ncat)
        lnl, lens, keys = ctx.score(aid, e, l, "full")
        fixed = ctx.score(aid, e, l, "fixed")[0]
        for k in (1, 3, 19, 37, 75, 151):
            lnl_k, lens_k, keys_k = ctx.score(aid, e[:k], l[:k], "full")
            np.testing.assert_array_equal(lnl_k, lnl[:k])
            np.testing.assert_array_equal(lens_k, lens[:k])
            np.testing.assert_array_equal(keys_k, keys[:k])
            np.testing.assert_array_equal(ctx.score(aid, e[:k], l[:k], "fixed")[0], fixed[:k])


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("n,sites,ncat", [(9, 120, 4), (12, 700, 1), (14, 1200, 4)])
def test_proposals_are_shape_independent(prec, n, sites, ncat):
    """The neighbours of one frontier tree, alone and in a round of many."""
    a, e, l = _case(n, sites, ncat, 40, 0.1)
    with pt.Context(precision=prec, table_log2=16) as ctx:
        aid = ctx.load_alignment(a.codes)
        ctx.set_model(aid, a.exch, a.freqs, 0.5, ncat)

        def props(k):
            ctx.reset_visited(aid)
            ctx.expand(aid, e[:k], l[:k], 0.0, 0.0)  # keeps nothing: proposals only
            p = ctx.last_proposals()
            return {(int(p["parent"][i]),) + tuple(int(x) for x in p["keys"][i]): (p["lnl"][i], *p["len5"][i])
                    for i in range(len(p["lnl"]))}
        many = props(40)
        for k in (1, 2, 5):
            few = props(k)
            both = set(few) & set(many)
            assert len(both) >= len(few) // 2  # the others have another proposer in the larger round
            assert all(few[x] == many[x] for x in both)


@pytest.mark.parametrize("P", [1545, 1555])
def test_noalloc_at_its_array_limit(P):
    """84 taxa in FP64: one tree's vectors fill the fixed array, so the sum-table has to fit in shared memory.
    Tolerance: P * 2^-52 * |lnL| of summation and about 1e3 * 2^-52 a site, below 1e-12 of |lnL|."""
    torch = pytest.importorskip("torch")
    n, dev = 84, torch.device("cuda", 0)
    tips = np.random.default_rng(P).integers(0, 4, (n, P)).astype(np.uint8)
    w = np.ones(P, np.int32)
    e, _ = synth.random_trees(n, 1, 3)
    l = np.full((1, 2 * n - 3), 0.1)
    exch, freqs = np.array([1.0, 2.0, 0.7, 1.1, 2.5, 1.0]), np.array([0.3, 0.2, 0.2, 0.3])
    want = oracle.Problem(tips, w, exch, freqs, 0.5, 4).loglik(e[0], l[0])
    cfg = pt.default_config()
    cfg.precision = pt.PREC_FP64
    t = [torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in (tips, w, e, l)]
    o_len, o_lnl = torch.empty_like(t[3]), torch.empty(1, dtype=torch.float64, device=dev)
    st = pt.score_noalloc(n, P, t[0].data_ptr(), t[1].data_ptr(), exch, freqs, 0.5, 4, 1, t[2].data_ptr(),
                          t[3].data_ptr(), o_len.data_ptr(), o_lnl.data_ptr(), mode="fixed",
                          stream=torch.cuda.current_stream().cuda_stream, cfg=cfg)
    assert st == 0
    torch.cuda.synchronize()
    np.testing.assert_allclose(o_lnl.item(), want, rtol=1e-12)
