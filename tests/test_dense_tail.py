"""The last rounds on a dense matrix: whole solves of graphs small enough to go
there at once, at the edges of its column groups, size and bound, against the
oracle."""
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


@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 64, 65, 96, 127, 160, 193, 223, 224, 225, 256])
@pytest.mark.parametrize("wmax", [1, 100])
def test_sizes(mc, n, wmax):
    for seed in range(3):
        solve(mc, graphgen.random_connected(n, 3 * n, seed=100 * n + seed, wmax=wmax))


@pytest.mark.parametrize("w", [(1 << 22) - 2, (1 << 22) - 1, 1 << 22, 1 << 28])
def test_bounds(mc, w):
    # a tree's edges and a cycle's halves at the largest bound taken, and past it
    g = graphgen.path_weights([w, w + 5, w, w + 9])
    solve(mc, g, w)
    half = w // 2
    solve(mc, graphgen.cycle(50, half), 2 * half)
    rng = np.random.default_rng(3)
    u, v = np.triu_indices(12, 1)
    solve(mc, graphgen.from_edges(12, u, v, rng.integers(w // 16, w // 11, size=len(u))))


def test_levels_and_shapes(mc):
    for level in range(5):
        for g in (graphgen.cycle(200, 3), graphgen.random_tree(180, 6), graphgen.two_cliques(60, 5),
                  graphgen.planted(3, block_n=100, avg_deg=30, cross=4)):
            solve(mc, g, pr_level=level)
            solve(mc, g, pr_level=level, seed=level + 9)
    two = graphgen.from_edges(30, list(range(14)) + list(range(15, 29)), list(range(1, 15)) + list(range(16, 30)))
    solve(mc, two, 0)
