"""Performance cases of the PT hot path: the calls a search program makes, over
the sizes it makes them at.

Every case simulates an alignment from its seed (paper_1811_11007_gb300.synth:
the model recipe of the benchmark and the tests), keeps a context with the
alignment and its model loaded -- what a search program holds -- and times one
pass of public calls:

  fixed   Context.score(..., "fixed"): log-likelihoods at given lengths, as for
          rescoring a sample of trees.
  full    Context.score(..., "full"): the visit, full branch-length optimisation.
  round   reset_visited + expand: one PT round on a frontier in host buffers.
  graph   reset_visited + set_frontier + run + next: the same round over several
          uneven alignments, replayed as a recorded CUDA graph.
  search  begin + expand until the frontier is empty + visited: a whole search.
  climb   hill_climb from perturbed topologies.

No visited table, frontier or tuned launch shape is carried from one pass to the
next; launch shapes are the library's defaults (no tuning).
"""
from __future__ import annotations

import math

import numpy as np

from paper_1811_11007_gb300 import pt, synth

ALPHA = 0.5      # Gamma shape of every GTR+G4 model, as in the benchmark
INIT = 0.1       # starting length of trees that were never optimised


def listed():
    return [
        # the smallest call: the log-likelihood of one tree, at the sizes of the paper's smaller datasets
        dict(name="fixed_1", kind="fixed", taxa=27, sites=2000, branch=0.05, trees=1, precision="mixed"),
        # rescoring a sample of trees (every tree of a search's result under one model)
        dict(name="fixed_256", kind="fixed", taxa=64, sites=1500, branch=0.05, trees=256, precision="mixed"),
        # optimising a handful of starting trees: how a search begins
        dict(name="full_8", kind="full", taxa=27, sites=2000, branch=0.05, trees=8, precision="mixed"),
        # the starting trees of the benchmark's large alignment
        dict(name="full_128x10000", kind="full", taxa=128, sites=10000, branch=0.02, trees=32, precision="mixed"),
        # one round of a search on a small alignment
        dict(name="round_27", kind="round", taxa=27, sites=2000, branch=0.05, frontier=48, threshold=10.0,
             precision="mixed", propose="five", prior=0.0),
        # one round on an alignment of middling size whose pattern count is near a CTA's shared memory
        dict(name="round_48", kind="round", taxa=48, sites=5000, branch=0.05, frontier=24, threshold=10.0,
             precision="mixed", propose="five", prior=0.0),
        # one round of the benchmark's workload
        dict(name="round_128x10000", kind="round", taxa=128, sites=10000, branch=0.02, frontier=24, threshold=15.0,
             precision="mixed", propose="five", prior=0.0),
        # the paper's default proposal (radius 0: the new branch only) under a branch-length prior
        dict(name="round_central_map", kind="round", taxa=41, sites=1201, branch=0.05, frontier=32, threshold=10.0,
             precision="mixed", propose="central", prior=10.0),
        # the FP64 path, which a user takes to check a result
        dict(name="round_fp64", kind="round", taxa=18, sites=900, branch=0.05, frontier=24, threshold=10.0,
             precision="fp64", propose="five", prior=0.0),
        # several uneven alignments at once, the graph replayed as a long search does
        dict(name="graph_4", kind="graph", shapes="20x300,33x1100,61x2501,100x5000", branch=0.05, frontier=12,
             threshold=10.0),
        # an exhaustive search of all 945 topologies on seven taxa (JC69, one rate, infinite threshold)
        dict(name="search_7", kind="search", taxa=7, sites=500, branch=0.1, precision="mixed"),
        # hill-climbs to the local maxima that seed a search
        dict(name="climb_8", kind="climb", taxa=27, sites=2000, branch=0.05, trees=8, moved=2, precision="mixed"),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fixed", "fixed", "full", "full", "round", "round", "round", "graph", "search", "climb"])
    branch = round(rng.uniform(0.02, 0.06), 3)
    precision = rng.choice(["mixed", "mixed", "mixed", "fp64"])
    taxa = _loguniform(rng, 8, 128)
    sites = _loguniform(rng, 200, 10000)
    size = taxa * sites
    if kind in ("fixed", "full"):
        most = 512 if kind == "fixed" else 64
        trees = _loguniform(rng, 1, max(1, min(most, (128 * 10000 * 32) // size)))
        if precision == "fp64":  # the FP64 rates are far lower: small problems only
            taxa, sites = min(taxa, 40), min(sites, 1500)
            trees = max(1, trees // 16)
        return dict(kind=kind, taxa=taxa, sites=sites, branch=branch, trees=trees, precision=precision)
    if kind == "round":
        if precision == "fp64":
            taxa, sites = min(taxa, 24), min(sites, 1200)
        front = _loguniform(rng, 1, max(1, min(96, (128 * 128 * 10000 * 24) // (taxa * taxa * sites))))
        if precision == "fp64":
            front = min(front, 16)
        return dict(kind="round", taxa=taxa, sites=sites, branch=branch, frontier=front,
                    threshold=round(rng.uniform(5.0, 15.0), 2), precision=precision,
                    propose=rng.choice(["five", "five", "central"]), prior=rng.choice([0.0, 0.0, 10.0]))
    if kind == "graph":
        shapes = ",".join("%dx%d" % (rng.randint(20, 100), _loguniform(rng, 300, 5000))
                          for _ in range(rng.randint(2, 6)))
        return dict(kind="graph", shapes=shapes, branch=branch, frontier=rng.randint(1, 12), threshold=10.0)
    if kind == "search":
        return dict(kind="search", taxa=rng.randint(5, 7), sites=_loguniform(rng, 200, 2000), branch=0.1,
                    precision=rng.choice(["mixed", "fp64"]))
    return dict(kind="climb", taxa=min(taxa, 48), sites=min(sites, 3000), branch=branch, trees=rng.randint(1, 12),
                moved=rng.randint(1, 3), precision="mixed")


# ---------------------------------------------------------------- inputs
def _seed(seed):
    return synth.SEED_BASE + 7919 * (int(seed) % (1 << 30))


def _alignment(taxa, sites, branch, seed, jc=False):
    """An alignment with its generating tree and model."""
    if jc:
        return synth.simulate(taxa, sites, seed, model="jc", alpha=None, mean_branch=branch)
    return synth.simulate(taxa, sites, seed, model="gtr", alpha=ALPHA, mean_branch=branch)


def _near_trees(a, taxa, count, moved, seed):
    """The generating topology with `moved` leaves reinserted, `count` times."""
    rng = np.random.default_rng(seed + 1)
    e = np.stack([synth.reinsert_leaves(a.tree_edges, taxa, moved, rng) for _ in range(count)])
    return np.ascontiguousarray(e, np.int32), rng


def _tree_inputs(case, seed):
    """Alignment, edges and lengths of a fixed / full / climb case."""
    s = _seed(seed)
    a = _alignment(case["taxa"], case["sites"], case["branch"], s)
    e, rng = _near_trees(a, case["taxa"], case["trees"], case.get("moved", 2), s)
    if case["kind"] == "fixed":  # lengths as a sample of trees has them
        l = rng.exponential(case["branch"], (case["trees"], 2 * case["taxa"] - 3)) + 1e-4
    else:
        l = np.full((case["trees"], 2 * case["taxa"] - 3), INIT)
    return a, e, l


def _context(case, a, jc=False, **kw):
    ctx = pt.Context(precision=case.get("precision", "mixed"), table_log2=kw.pop("table_log2", 22), **kw)
    aid = ctx.load_alignment(a.codes)
    ctx.set_model(aid, a.exch, a.freqs, 1.0 if jc else ALPHA, 1 if jc else 4)
    return ctx, aid


def _frontier(ctx, aid, a, taxa, most, threshold):
    """The frontier of a search from the generating topology, at most `most` trees of it, and lmax."""
    lmax, front = ctx.begin(aid, a.tree_edges[None], np.full((1, 2 * taxa - 3), INIT), threshold)
    for _ in range(4):
        if len(front["edges"]) >= most:
            break
        lm, nxt = ctx.expand(aid, front["edges"], front["lengths"], threshold, lmax)
        if len(nxt["edges"]) <= len(front["edges"]):
            break
        lmax, front = lm, nxt
    return lmax, front["edges"][:most].copy(), front["lengths"][:most].copy()


def _room(taxa, frontier):
    """Where a program keeps the next frontier: room for every neighbour of `frontier` trees."""
    cap, E = frontier * 2 * (taxa - 3), 2 * taxa - 3
    return {"edges": np.zeros((cap, E, 2), np.int32), "lengths": np.zeros((cap, E)), "lnl": np.zeros(cap),
            "keys": np.zeros((cap, 2), np.int64), "count": 0}


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind in ("fixed", "full", "climb"):
        a, st["e"], st["l"] = _tree_inputs(case, seed)
        st["ctx"], st["aid"] = _context(case, a)
    elif kind == "round":
        a = _alignment(case["taxa"], case["sites"], case["branch"], _seed(seed))
        st["ctx"], st["aid"] = _context(case, a, propose=case["propose"], branch_prior_rate=case["prior"])
        st["lmax"], st["e"], st["l"] = _frontier(st["ctx"], st["aid"], a, case["taxa"], case["frontier"],
                                                 case["threshold"])
        st["next"] = _room(case["taxa"], case["frontier"])
    elif kind == "graph":
        st["ctx"] = ctx = pt.Context(precision="mixed", table_log2=18)
        st["parts"], st["next"] = [], []
        for k, shape in enumerate(case["shapes"].split(",")):
            n, sites = (int(x) for x in shape.split("x"))
            a = _alignment(n, sites, case["branch"], _seed(seed) + 101 * k)
            aid = ctx.load_alignment(a.codes)
            ctx.set_model(aid, a.exch, a.freqs, ALPHA, 4)
            st["parts"].append((aid,) + _frontier(ctx, aid, a, n, case["frontier"], case["threshold"]))
            st["next"].append(_room(n, case["frontier"]))
        na = len(st["parts"])
        st["graph"] = ctx.graph([p[0] for p in st["parts"]], [case["frontier"]] * na, [case["threshold"]] * na)
    else:
        s = _seed(seed)
        a = _alignment(case["taxa"], case["sites"], case["branch"], s, jc=True)
        st["ctx"], st["aid"] = _context(case, a, jc=True, table_log2=14)
        st["e"], st["l"] = synth.random_trees(case["taxa"], 1, s + 1, INIT)
    return st


def _keys(k):
    return np.ascontiguousarray(k, np.uint64).view(np.int64)


def _keep(room, f):
    """The next frontier into the program's own arrays."""
    k = room["count"] = len(f["edges"])
    for name in ("edges", "lengths", "lnl"):
        room[name][:k] = f[name]
    room["keys"][:k] = _keys(f["keys"])
    return room


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind = case["kind"]
    if kind in ("fixed", "full"):
        lnl, lens, keys = ctx.score(st["aid"], st["e"], st["l"], kind)
        return {"lnl": lnl, "lengths": lens, "keys": _keys(keys)}
    if kind == "round":
        ctx.reset_visited(st["aid"])
        lmax, nxt = ctx.expand(st["aid"], st["e"], st["l"], case["threshold"], st["lmax"])
        return {"lmax": lmax, "next": _keep(st["next"], nxt)}
    if kind == "graph":
        g = st["graph"]
        for k, (aid, lmax, e, l) in enumerate(st["parts"]):
            ctx.reset_visited(aid)
            g.set_frontier(k, e, l)
        lm, _ = g.run([len(p[2]) for p in st["parts"]], [p[1] for p in st["parts"]])
        return {"lmax": np.array(lm), "next": [_keep(room, g.next(k)) for k, room in enumerate(st["next"])]}
    if kind == "search":
        lmax, front = ctx.begin(st["aid"], st["e"], st["l"], math.inf)
        while len(front["edges"]):
            lmax, front = ctx.expand(st["aid"], front["edges"], front["lengths"], math.inf, lmax)
        vis = ctx.visited(st["aid"])
        order = np.lexsort((vis["keys"][:, 0], vis["keys"][:, 1]))  # the table's order is not part of the result
        return {"lmax": lmax, "keys": _keys(vis["keys"][order]), "status": vis["status"][order],
                "lnl": vis["lnl"][order]}
    r = ctx.hill_climb(st["aid"], st["e"], st["l"])
    return {"edges": r["edges"], "lengths": r["lengths"], "lnl": r["lnl"], "keys": _keys(r["keys"]),
            "moves": r["moves"]}


# ---------------------------------------------------------------- work
# Flops per site pattern of one 4-state, C-category vector: a transition-matrix
# product 28 C, a combination of two children 60 C, a branch's sum-table (two
# eigenbasis changes, products) 100 C, one evaluation of L, L', L'' 24 C.
def _patterns(sites):
    return max(1, int(0.5 * sites))  # half of the columns are repeats at these branch lengths


def work(case):
    kind = case["kind"]
    shapes = ([tuple(int(v) for v in x.split("x")) for x in case["shapes"].split(",")] if kind == "graph"
              else [(case["taxa"], case["sites"])])
    C = 1 if kind == "search" else 4
    total = {"bytes": 0, "flops": 0}
    for n, sites in shapes:
        P, E = _patterns(sites), 2 * n - 3
        tree = E * 16 + 24                                     # edges, lengths, score and key
        prune = (n - 2) * P * 60 * C + P * 36 * C              # one pruning pass
        sweep = E * P * (60 + 100 + 2 * 24) * C + (n - 2) * P * 60 * C  # two evaluations per branch
        full = prune + 2 * sweep                               # one sweep that moves, one that confirms
        nb = 1 if case.get("propose") == "central" else 5
        prop = 2 * nb * P * (2 * 60 + 100 + 2 * 24) * C        # the same on the proposal's branches
        if kind == "fixed":
            trees, flops = case["trees"], case["trees"] * prune
        elif kind == "full":
            trees, flops = case["trees"], case["trees"] * full
        elif kind == "climb":  # one neighbourhood per move and the one that ends the climb
            steps = case["moved"] + 1
            trees, flops = case["trees"], case["trees"] * (full + steps * (2 * prune + 2 * (n - 3) * prop + full))
        elif kind == "search":
            trees = math.prod(range(1, 2 * n - 4, 2))          # every topology, each optimised once
            flops = trees * (full + prop)
        else:  # a round: the frontier's vectors, its neighbours (half of them shared), as many visits as trees
            trees = case["frontier"]
            flops = trees * (2 * prune + (n - 3) * prop + full)
        total["bytes"] += 2 * trees * tree + n * P + 4 * P
        total["flops"] += flops
    return total


# ---------------------------------------------------------------- the same in 64 bits, plainly
class _Plain:
    """GTR+Gamma likelihoods and the full branch optimisation in numpy float64."""

    def __init__(self, a, n, ncat, rates):
        cols, w = np.unique(a.codes.T, axis=0, return_counts=True)
        self.n, self.w, self.C, self.rates = n, w.astype(np.float64), ncat, rates
        tip = np.eye(4)
        self.tips = [np.where((cols[:, t] >= 4)[:, None], 1.0, tip[np.minimum(cols[:, t], 3)]) for t in range(n)]
        iu = [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]
        S = np.zeros((4, 4))
        for k, (i, j) in enumerate(iu):
            S[i, j] = S[j, i] = a.exch[k]
        pi = np.asarray(a.freqs, np.float64) / np.sum(a.freqs)
        Q = S * pi[None]
        np.fill_diagonal(Q, -Q.sum(1))
        Q /= -float(np.sum(pi * np.diag(Q)))
        d = np.sqrt(pi)
        lam, R = np.linalg.eigh((d[:, None] * Q / d[None] + (d[:, None] * Q / d[None]).T) / 2)
        self.pi, self.lam = pi, lam
        self.L, self.Ri = R / d[:, None], R.T * d[None]   # P(t) = L exp(lam t) Ri

    def P(self, t):
        return np.stack([(self.L * np.exp(self.lam * r * t)[None]) @ self.Ri for r in self.rates])

    def vec(self, v):
        """A tip as [C][patterns][4], and its (zero) log scales."""
        return np.broadcast_to(self.tips[v], (self.C,) + self.tips[v].shape), np.zeros(len(self.w))

    def join(self, t0, a, t1, b):
        y = (a[0] @ self.P(t0).transpose(0, 2, 1)) * (b[0] @ self.P(t1).transpose(0, 2, 1))
        m = y.max((0, 2))
        return y / m[None, :, None], a[1] + b[1] + np.log(m)

    def root(self, edges, lengths):
        """Children (smallest taxon first), edge index to the parent and first inner node, rooted at leaf 0."""
        n, adj = self.n, {}
        for k, (x, y) in enumerate(edges):
            adj.setdefault(int(x), []).append((int(y), k))
            adj.setdefault(int(y), []).append((int(x), k))
        top = adj[0][0][0]
        kids, eid, least, order, stack = {}, {top: adj[0][0][1]}, {}, [], [(top, 0)]
        while stack:
            v, par = stack.pop()
            order.append(v)
            kids[v] = [c for c, _ in adj[v] if c != par]
            for c, k in adj[v]:
                if c != par:
                    eid[c] = k
                    stack.append((c, v))
        for v in reversed(order):
            least[v] = v if v < n else min(least[c] for c in kids[v])
            kids[v].sort(key=lambda c: least[c])
        return top, kids, eid, order

    def down(self, lengths, kids, eid, order):
        D = {}
        for v in reversed(order):
            D[v] = self.vec(v) if v < self.n else self.join(lengths[eid[kids[v][0]]], D[kids[v][0]],
                                                            lengths[eid[kids[v][1]]], D[kids[v][1]])
        return D

    def across(self, X, Y, t):
        site = np.einsum("i,cpi,cpi->p", self.pi, X[0], Y[0] @ self.P(t).transpose(0, 2, 1)) / self.C
        return float(self.w @ (np.log(site) + X[1] + Y[1]))

    def lnl(self, edges, lengths):
        top, kids, eid, order = self.root(edges, lengths)
        return self.across(self.vec(0), self.down(lengths, kids, eid, order)[top], lengths[eid[top]])

    def solve(self, X, Y, t, cfg):
        """One safeguarded Newton solve of the length between X and Y."""
        s = (X[0] * self.pi @ self.L) * (Y[0] @ self.Ri.T)       # [C][p][k]: coefficients of exp(lam_k r t)
        lr = np.outer(self.rates, self.lam)
        lo, hi = cfg.tmin, cfg.tmax
        t = min(max(t, lo), hi)
        for _ in range(cfg.newton_maxit):
            e = np.exp(lr * t)
            f, f1, f2 = (np.einsum("cpk,ck->p", s, e * lr ** k) for k in range(3))
            g = f1 / f
            d1, d2 = float(self.w @ g), float(self.w @ (f2 / f - g * g))
            if d1 == 0:
                break
            if d1 > 0:
                lo = t
            else:
                hi = t
            new = t - d1 / d2 if d2 < 0 else -1.0
            if not lo < new < hi:
                new = math.sqrt(lo * hi)
            moved, t = abs(new - t), new
            if moved <= cfg.newton_tol:
                break
        return t

    def optimise(self, edges, lengths, cfg):
        """Sweeps over all branches in pre-order until none moves by more than sweep_tol."""
        top, kids, eid, order = self.root(edges, lengths)
        t = np.array(lengths, np.float64)
        D = self.down(t, kids, eid, order)
        for _ in range(cfg.full_max_sweeps):
            moved = 0.0
            todo = [(top, self.vec(0))]
            while todo:
                v, X = todo.pop()
                if X is None:  # the subtree of v is done
                    c0, c1 = kids[v]
                    D[v] = self.join(t[eid[c0]], D[c0], t[eid[c1]], D[c1])
                    continue
                if not isinstance(X[0], np.ndarray):  # (parent, sibling, the vector above the parent)
                    u, sib, up = X
                    X = self.join(t[eid[sib]], D[sib], t[eid[u]], up)
                new = self.solve(X, D[v], t[eid[v]], cfg)
                moved = max(moved, abs(new - t[eid[v]]))
                t[eid[v]] = new
                if v >= self.n:
                    c0, c1 = kids[v]
                    todo += [(v, None), (c1, (v, c0, X)), (c0, (v, c1, X))]
            if moved <= cfg.sweep_tol:
                break
        return t, self.lnl(edges, t)


def _gamma_rates(alpha, ncat):
    """Mean rates of equal-probability categories of Gamma(alpha, alpha): bisection on the regularised
    incomplete gamma function, by its power series."""
    if ncat == 1:
        return np.ones(1)

    def P(s, x):
        term = tot = 1.0 / s
        k = 0
        while term > tot * 1e-18:
            k += 1
            term *= x / (s + k)
            tot += term
        return tot * math.exp(s * math.log(x) - x - math.lgamma(s)) if x > 0 else 0.0

    cum = [0.0]
    for k in range(1, ncat):
        lo, hi = 0.0, 60.0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if P(alpha, mid) < k / ncat else (lo, mid)
        cum.append(P(alpha + 1, 0.5 * (lo + hi)))
    r = ncat * np.diff(cum + [1.0])
    return r * ncat / r.sum()


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("fixed", "full"):
        return None  # hundreds to thousands of optimisations: minutes in plain numpy
    cost = case["trees"] * case["taxa"] * case["sites"]
    if cost > (4e7 if kind == "fixed" else 1e6):
        return None
    a, e, l = _tree_inputs(case, seed)
    m = _Plain(a, case["taxa"], 4, _gamma_rates(ALPHA, 4))
    if kind == "fixed":
        return {"lnl": np.array([m.lnl(x, y) for x, y in zip(e, l)]), "lengths": l, "keys": None}
    cfg = pt.Config(tmin=1e-6, tmax=100.0, newton_tol=1e-8, sweep_tol=1e-6, newton_maxit=50, full_max_sweeps=64)
    got = [m.optimise(x, y, cfg) for x, y in zip(e, l)]
    return {"lnl": np.array([g[1] for g in got]), "lengths": np.stack([g[0] for g in got]), "keys": None}
