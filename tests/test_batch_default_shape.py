"""The batched solver's default shape and its late PR tests: every lambda
against the oracle at the sizes where the default changes, and on graphs that
only the PR tests finish in few rounds."""
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
    m.batch_set_shape(-1)
    return m


def concatenate(graphs):
    rp = np.concatenate([g[0] for g in graphs]).astype(np.int32)
    col = np.concatenate([g[1] for g in graphs]).astype(np.int32)
    w = np.concatenate([g[2] for g in graphs]).astype(np.int32)
    voff = np.concatenate([[0], np.cumsum([len(g[0]) - 1 for g in graphs])]).astype(np.int64)
    aoff = np.concatenate([[0], np.cumsum([len(g[1]) for g in graphs])]).astype(np.int64)
    return rp, col, w, voff, aoff


def check(mc, b):
    lam, bits, boff, _ = mc.batch_min_cut(*b, bitmaps=True)
    for k in range(len(lam)):
        g = graphgen.batch_graph(b, k)
        n = len(g[0]) - 1
        side = mc.bitmap_to_side(bits[boff[k]:boff[k + 1]], n)
        assert lam[k] == oracle.noi(*g)[0]
        assert side[0] == 0 and 0 < side.sum() < n and oracle.cut_weight(*g, side) == lam[k]


@pytest.mark.parametrize("nmax", [510, 511, 1022, 1023, 2046, 2049])
@pytest.mark.parametrize("graphs", [5, 700])
def test_sizes_at_the_shapes_edges(mc, nmax, graphs):
    small = [graphgen.batch_graph(graphgen.batch(7, 1, 12, 12, 4, 6, 9), 0)] * (graphs - 2)
    big = [graphgen.batch_graph(graphgen.batch(nmax + k, 1, nmax, nmax, 6, 6, 100), 0) for k in range(2)]
    check(mc, concatenate(big + small))


def test_paths_and_cycles(mc):
    rng = np.random.default_rng(5)
    graphs = [graphgen.cycle(n, w) for n, w in ((3, 1), (64, 2), (999, 1), (2000, 7))]
    graphs += [graphgen.path_weights(rng.integers(1, 50, size=n)) for n in (2, 31, 1500)]
    graphs += [graphgen.random_tree(900, 4), graphgen.two_cliques(30, 4), graphgen.complete(40, 3)]
    check(mc, concatenate(graphs))
