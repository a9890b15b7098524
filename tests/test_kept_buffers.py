"""A graph built into the buffers of a larger one destroyed before it goes
through the same rounds as in buffers of its own.  One vertex of small degree
beside random ones of heavy weights: the forests its bound asks for unite all but
that vertex where they fit, and they do not fit a graph's own buffers."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _heavy(n, deg, seed):
    rng = np.random.default_rng(seed)
    m = n * deg // 2
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    key = np.unique((np.minimum(u, v) * n + np.maximum(u, v))[u != v])
    u, v = np.concatenate([key // n, np.full(4, n)]), np.concatenate([key % n, rng.permutation(n)[:4]])
    return graphgen.from_edges(n + 1, u, v, rng.integers(25, 31, len(u)))


def test_rounds_do_not_depend_on_the_graph_before():
    import paper_1808_05458_gb300 as mc
    small, large = _heavy(3000, 40, 1), _heavy(30000, 80, 2)
    lam = oracle.noi(*small)[0]
    assert lam * 3001 > 2 * len(small[1])  # words the forests take, and the buffers hold
    scans = []
    # one takes the buffers kept from whatever was there, so the next gets its own
    with mc.Graph(*small), mc.Graph(*small) as own:
        scans.append(own.min_cut().stats["scan_launches"] > 0)
    with mc.Graph(*large):
        pass
    with mc.Graph(*small) as kept:
        r = kept.min_cut()
    scans.append(r.stats["scan_launches"] > 0)
    assert r.lam == lam == oracle.cut_weight(*small, r.side(3001))
    assert scans[0] == scans[1]
