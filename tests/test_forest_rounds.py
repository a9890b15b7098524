"""Rounds of connectivity certificates by forest packing, against the oracle.

The packing is the solver's way on graphs that are not clustered, so its
blocks are checked through whole solves: lambda equal to the oracle's, the
returned side re-weighed.  Sizes lie at the edges of the kernels' tiles (32
vertices a block, 65536 between the two starting passes), with the small-graph
finish off where the rounds themselves should reach the end.
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


def random_graph(seed, n, deg, wmax):
    return graphgen.batch_graph(graphgen.batch(seed, 1, n, n, deg, deg, wmax), 0)


def test_tiny_graphs_by_rounds_alone(mc):
    rng = np.random.default_rng(31)
    for i in range(150):
        n = int(rng.integers(2, 15))
        g = graphgen.random_gnp(n, float(rng.uniform(0.3, 1.0)), seed=i, wmax=int(rng.integers(1, 7)))
        if len(g[1]) == 0:
            continue
        solve(mc, g, oracle.brute_force(*g)[0], tail_vertices=-1)


@pytest.mark.parametrize("n", [31, 32, 33, 255, 257, 4097, 65535, 65536, 65569])
@pytest.mark.parametrize("wmax", [1, 4])
def test_random_graphs_at_tile_edges(mc, n, wmax):
    solve(mc, random_graph(n + wmax, n, 12, wmax), tail_vertices=-1)


@pytest.mark.parametrize("wmax", [30, 400, 5000])
def test_heavy_weights(mc, wmax):
    # bounds from a few hundred (still packed) to past the packing's limits
    solve(mc, random_graph(wmax, 3000, 40, wmax), tail_vertices=-1)


@pytest.mark.parametrize("k", [10, 50])
def test_skewed_cores(mc, k):
    g = graphgen.rmat_kcore(5, 15, k=k)
    solve(mc, g)
    solve(mc, g, bound=mc.MC_BOUND_LP)


@pytest.mark.parametrize("cross", [0, 1, 5])
def test_cut_between_two_blocks(mc, cross):
    # both blocks find representatives of their own; with no edge between
    # them lambda is 0
    g = graphgen.planted(cross + 1, block_n=3000, avg_deg=40, cross=cross)
    r = solve(mc, g)
    assert r.lam == cross


def test_sparse_graphs_fall_back(mc):
    # fewer edges than the forests hold: the packing unites little, the scans go on
    for seed in range(4):
        solve(mc, random_graph(seed, 2000, 4, 100), tail_vertices=-1)
    solve(mc, graphgen.random_tree(1500, 3), tail_vertices=-1)


def test_scan_options_keep_the_scans(mc):
    g = random_graph(9, 5000, 16, 1)
    lam = oracle.noi(*g)[0]
    for opt in ({}, dict(visits=2), dict(region_budget=64), dict(scans_per_round=64), dict(pq_order=mc.MC_PQ_FIFO)):
        r = solve(mc, g, lam, **opt)
        assert (r.stats["scan_launches"] == 0) == (opt == {})
