"""The warps' part of a batch nobody tuned: its shape at the sizes where the
default changes, and the PR tests that run after a poor round only.  Every
graph's rows are in falling order, which the block-per-graph solver leaves to
the warps (they sort them), so that each is solved by these; lambda and the
side's weight against the oracle."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import paper_1808_05458_gb300 as m
    m.load_library()
    m.batch_set_shape(-1)
    return m


def _falling(g):
    rp, col, w = g
    row = np.repeat(np.arange(len(rp) - 1), np.diff(rp))
    o = np.lexsort((-col.astype(np.int64), row))
    return rp, col[o], w[o]


def _check(mc, graphs):
    gs = [_falling(g) for g in graphs]
    vo = np.concatenate([[0], np.cumsum([len(g[0]) - 1 for g in gs])])
    ao = np.concatenate([[0], np.cumsum([len(g[1]) for g in gs])])
    lam, bits, bo, _ = mc.batch_min_cut(*(np.concatenate([g[k] for g in gs]).astype(np.int32) for k in range(3)),
                                        vo, ao, bitmaps=True)
    for k, g in enumerate(graphs):
        n = len(g[0]) - 1
        side = mc.bitmap_to_side(bits[bo[k]:bo[k + 1]], n)
        assert lam[k] == oracle.noi(*g)[0]
        assert side[0] == 0 and 0 < side.sum() < n and oracle.cut_weight(*g, side) == lam[k]


@pytest.mark.parametrize("nmax", [254, 255, 510, 511, 1022, 1023, 2046, 2047])
@pytest.mark.parametrize("small", [3, 700])
def test_sizes_at_the_shapes_edges(mc, nmax, small):
    one = graphgen.batch_graph(graphgen.batch(7, 1, 12, 12, 4, 6, 9), 0)
    big = [graphgen.batch_graph(graphgen.batch(nmax + k, 1, nmax, nmax, 6, 6, 100), 0) for k in range(2)]
    _check(mc, big + [one] * small)


def test_poor_rounds(mc):
    rng = np.random.default_rng(5)
    graphs = [graphgen.cycle(n, w) for n, w in ((3, 1), (64, 2), (500, 3), (999, 1), (2000, 7))]
    graphs += [graphgen.path_weights(rng.integers(1, 50, size=n)) for n in (2, 31, 300, 1500)]
    graphs += [graphgen.random_tree(900, 4), graphgen.two_cliques(30, 4), graphgen.complete(40, 3)]
    _check(mc, graphs)
    for most in (510, 1022):  # and enough of them for each of the other shapes
        fit = [g for g in graphs if len(g[0]) - 1 <= most]
        _check(mc, fit * (700 // len(fit) + 1))
