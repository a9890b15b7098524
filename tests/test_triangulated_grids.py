"""Graphs with triangles in two wedges of five: triangulated grids (lambda = 2 at
two corners) and small worlds go to the triangle tests, which leave little for a
second round.  Closed form and the oracle."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _grid(a, b, seed):
    i = np.arange(a * b).reshape(a, b)
    u = np.concatenate([i[:-1].ravel(), i[:, :-1].ravel(), i[:-1, :-1].ravel()])
    v = np.concatenate([i[1:].ravel(), i[:, 1:].ravel(), i[1:, 1:].ravel()])
    p = np.random.default_rng(seed).permutation(a * b)
    return graphgen.from_edges(a * b, p[u], p[v])


def _small_world(n, k, share, seed):
    rng = np.random.default_rng(seed)
    u = np.repeat(np.arange(n), k)
    v = (u + np.tile(np.arange(1, k + 1), n)) % n
    v = np.where(rng.random(len(u)) < share, rng.integers(0, n, len(u)), v)
    key = np.unique((np.minimum(u, v) * n + np.maximum(u, v))[u != v])
    return graphgen.from_edges(n, key // n, key % n)


@pytest.mark.parametrize("a,b", [(20, 31), (64, 64), (128, 128), (333, 97)])
def test_grids(a, b):
    import paper_1808_05458_gb300 as mc
    g = _grid(a, b, a)
    with mc.Graph(*g) as G:
        r = G.min_cut()
    assert r.lam == 2 == oracle.cut_weight(*g, r.side(a * b))
    assert r.stats["rounds"] <= 2 and r.stats["scan_launches"] == 0


@pytest.mark.parametrize("k,share", [(3, 0.05), (4, 0.1), (4, 0.2), (8, 0.15)])
def test_small_worlds(k, share):
    import paper_1808_05458_gb300 as mc
    for seed in range(3):
        g = _small_world(6000, k, share, seed)
        with mc.Graph(*g) as G:
            r = G.min_cut(mc.options(tail_vertices=-1))
        assert r.lam == oracle.noi(*g)[0] == oracle.cut_weight(*g, r.side(6000))
