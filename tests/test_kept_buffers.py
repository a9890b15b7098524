"""A graph built into the buffers of a larger one destroyed before it goes
through the same rounds as in buffers of its own.  One vertex of small degree
beside random ones of heavy weights: the forests its bound asks for do not fit a
graph's own buffers, the scans unite nothing and one full scan nearly all; packed
in larger buffers the forests unite a few vertices a round before that."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _heavy(n, deg, low, seed):
    rng = np.random.default_rng(seed)
    m = n * deg // 2
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    key = np.unique((np.minimum(u, v) * n + np.maximum(u, v))[u != v])
    u, v = np.concatenate([key // n, np.full(low, n)]), np.concatenate([key % n, rng.permutation(n)[:low]])
    return graphgen.from_edges(n + 1, u, v, rng.integers(10, 12, len(u)))


def test_rounds_do_not_depend_on_the_graph_before():
    import paper_1808_05458_gb300 as mc
    small, large = _heavy(6000, 30, 7, 1), _heavy(30000, 80, 7, 2)
    lam = oracle.noi(*small)[0]
    assert lam * 6001 > 2 * len(small[1])  # words the forests take, and the buffers hold

    def rounds(G):
        return {G.min_cut().stats["rounds"] for _ in range(8)}

    # one takes the buffers kept from whatever was there, so the next gets its own
    with mc.Graph(*small), mc.Graph(*small) as own:
        want = rounds(own)
    with mc.Graph(*large):
        pass
    with mc.Graph(*small) as kept:
        got = rounds(kept)
        r = kept.min_cut()
    assert r.lam == lam == oracle.cut_weight(*small, r.side(6001))
    assert got == want
