"""Cycles and chains in the block-per-graph batched solver, where the packing
unites little and the rule for degree 2 goes on: equal weights and one that
differs, chains between hubs, numbered in order and at random, with the rule and
without.  Exact."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _shuffled(g, seed):
    n = len(g[0]) - 1
    p = np.random.default_rng(seed).permutation(n)
    u = np.repeat(np.arange(n), np.diff(g[0]))
    k = u < g[1]
    return graphgen.from_edges(n, p[u[k]], p[g[1][k]], g[2][k])


def _graphs():
    rng = np.random.default_rng(2)
    out = [graphgen.cycle(n, w) for n, w in ((3, 1), (4, 5), (33, 1), (64, 2), (65, 3), (500, 1), (1001, 7), (2048, 1))]
    for n in (40, 300, 1500):
        i = np.arange(n)
        w = np.full(n, 4)
        w[n // 3] = 3
        out.append(graphgen.from_edges(n, i, (i + 1) % n, w))
        hub = np.concatenate([i, [0, n // 4]]), np.concatenate([(i + 1) % n, [n // 2, 3 * n // 4]])
        out.append(graphgen.from_edges(n, *hub, rng.integers(1, 3, n + 2)))
        out.append(graphgen.from_edges(n, *hub, np.full(n + 2, 2)))
        # a wheel of long spokes
        k = n // 10
        u = np.concatenate([np.arange(1, n), np.arange(1, n, k)])
        v = np.concatenate([np.where(np.arange(1, n) % k == 0, 0, np.arange(2, n + 1) % n), np.zeros(len(range(1, n, k)), int)])
        out.append(graphgen.from_edges(n, u, v, np.full(len(u), 2)))
    return out + [_shuffled(g, k) for k, g in enumerate(out)]


@pytest.mark.parametrize("level", [0, 1, 2, 4])
def test_cycles_and_chains(level):
    import paper_1808_05458_gb300 as mc
    mc.batch_set_shape(-1)
    graphs = _graphs()
    vo = np.concatenate([[0], np.cumsum([len(g[0]) - 1 for g in graphs])])
    ao = np.concatenate([[0], np.cumsum([len(g[1]) for g in graphs])])
    lam, bits, bo, _ = mc.batch_min_cut(*(np.concatenate([g[k] for g in graphs]).astype(np.int32) for k in range(3)),
                                        vo, ao, mc.options(pr_level=level), bitmaps=True)
    for k, g in enumerate(graphs):
        side = mc.bitmap_to_side(bits[bo[k]:bo[k + 1]], len(g[0]) - 1)
        assert lam[k] == oracle.noi(*g)[0] == oracle.cut_weight(*g, side)
        assert side[0] == 0 and 0 < side.sum() < len(g[0]) - 1
