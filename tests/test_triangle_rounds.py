"""Rounds of triangle tests on clustered graphs, against the oracle.

The tests are the solver's first round where most wedges are closed; they are
checked through whole solves, with the small-graph finish off where the rounds
should reach the end by themselves.
"""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import torch
    assert torch.cuda.is_available()
    import paper_1808_05458_gb300 as m
    m.load_library()
    return m


def solve(mc, g, lam=None, **opt):
    n = len(g[0]) - 1
    with mc.Graph(*g) as G:
        r = G.min_cut(mc.options(**opt))
    if lam is None:
        lam = oracle.noi(*g)[0]
    side = r.side(n)
    assert r.lam == lam
    assert side[0] == 0 and 0 < side.sum() < n
    assert oracle.cut_weight(*g, side) == lam
    return r


def ring_lattice(n, k, seed=0, wmax=1):
    """Every vertex joined to its k nearest on either side of a ring; ids shuffled."""
    rng = np.random.default_rng(seed)
    perm = rng.permutation(n)
    u = np.repeat(np.arange(n), k)
    v = (u + np.tile(np.arange(1, k + 1), n)) % n
    return graphgen.from_edges(n, perm[u], perm[v], rng.integers(1, wmax + 1, size=n * k))


def ring_of_cliques(cliques, size, joins, seed=0):
    """Cliques on a ring, `joins` unit edges from each to the next: lambda = 2 * joins."""
    rng = np.random.default_rng(seed)
    iu, ju = np.triu_indices(size, 1)
    base = np.arange(cliques)[:, None] * size
    u, v = (base + iu).ravel(), (base + ju).ravel()
    for c in range(cliques):
        u = np.concatenate([u, c * size + rng.permutation(size)[:joins]])
        v = np.concatenate([v, (c + 1) % cliques * size + rng.permutation(size)[:joins]])
    return graphgen.from_edges(cliques * size, u, v)


@pytest.mark.parametrize("n", [17, 31, 32, 33, 255, 257, 4096, 20011])
@pytest.mark.parametrize("wmax", [1, 5])
def test_ring_lattices(mc, n, wmax):
    solve(mc, ring_lattice(n, 4, seed=n, wmax=wmax), tail_vertices=-1)


@pytest.mark.parametrize("joins", [1, 2, 3])
def test_rings_of_cliques(mc, joins):
    solve(mc, ring_of_cliques(60, 12, joins), 2 * joins, tail_vertices=-1)
    solve(mc, ring_of_cliques(60, 12, joins), 2 * joins, approx_milli=500, tail_vertices=-1)


@pytest.mark.parametrize("n,deg", [(2000, 8.0), (5000, 16.0), (30011, 24.0), (20000, 64.0), (6000, 200.0)])
def test_hyperbolic(mc, n, deg):
    g = graphgen.rhg(7, n, deg)
    solve(mc, g)
    solve(mc, g, bound=mc.MC_BOUND_LP)


@pytest.mark.parametrize("wmax", [3, 1000, 1 << 22])
def test_weighted_hyperbolic(mc, wmax):
    # the largest weights put the bound past the tests' limit
    rp, col, _ = graphgen.rhg(3, 4000, 24.0)
    n = len(rp) - 1
    src = np.repeat(np.arange(n), np.diff(rp)).astype(np.int64)
    lo, hi = np.minimum(src, col), np.maximum(src, col)
    w = 1 + ((lo * 2654435761 + hi * 40503) % wmax)
    solve(mc, (rp, col, w.astype(np.int32)), tail_vertices=-1)


def test_cut_between_hyperbolic_blocks(mc):
    for cross in (1, 4):
        r = solve(mc, graphgen.planted_rhg(cross, 5000, 64.0, cross=cross), cross)
        assert r.stats["scan_launches"] == 0


def test_lower_levels_and_scan_options(mc):
    g = graphgen.rhg(2, 8000, 24.0)
    lam = oracle.noi(*g)[0]
    for opt in (dict(pr_level=0), dict(pr_level=3), dict(visits=2), dict(region_budget=64)):
        assert solve(mc, g, lam, **opt).stats["scan_launches"] > 0


def test_trusted_rows_without_mirrors(mc):
    # rows of one rank only: not symmetric, contracted arc by arc
    rp, col, w = graphgen.rhg(2, 3000, 24.0)
    n = len(rp) - 1
    keep = np.arange(len(col)) < rp[n // 3]
    rp2 = np.minimum(rp, rp[n // 3]).astype(np.int32)
    lab = (np.arange(n) // 5).astype(np.int32)
    nc = int(lab.max()) + 1
    with mc.Graph(rp2, col[keep], w[keep], trust=True) as G:
        out = G.contract(lab, nc)
    src = np.repeat(np.arange(n), np.diff(rp2))
    a, b = lab[src], lab[col[keep]]
    M = np.zeros((nc, nc), dtype=np.int64)
    np.add.at(M, (a[a != b], b[a != b]), w[keep][a != b])
    r, c = np.nonzero(M)
    assert (out[1] == c).all() and (out[2] == M[r, c]).all()
    assert (out[0] == np.concatenate([[0], np.cumsum(np.bincount(r, minlength=nc))])).all()
