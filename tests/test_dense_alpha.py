"""Cuts that only a scan's alpha finds on the dense matrix: the r of every
popped vertex goes into alpha, and it is another lane's, so a value that is one
pop old gives a wrong lambda.  Two blocks of a few hundred edges joined by less
than the minimum degree, at every number of column groups; exact."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _joined(half, cross, wmax, seed):
    rng = np.random.default_rng(seed)
    iu, iv = np.triu_indices(half, 1)
    keep = rng.random(len(iu)) < 0.8
    u, v = np.concatenate([iu[keep], iu[keep] + half]), np.concatenate([iv[keep], iv[keep] + half])
    w = rng.integers(1, wmax + 1, len(u))
    c = rng.permutation(half)[:cross]
    u, v, w = np.concatenate([u, c]), np.concatenate([v, c + half]), np.concatenate([w, np.ones(cross, int)])
    p = rng.permutation(2 * half)
    return graphgen.from_edges(2 * half, p[u], p[v], w)


@pytest.mark.parametrize("n", [16, 32, 34, 64, 66, 96, 98, 130, 162, 194, 224])
@pytest.mark.parametrize("wmax", [1, 50])
def test_alpha_of_every_pop(n, wmax):
    import paper_1808_05458_gb300 as mc
    for seed in range(6):
        g = _joined(n // 2, 2, wmax, 31 * n + seed)
        with mc.Graph(*g) as G:
            for s in range(4):
                r = G.min_cut(mc.options(seed=s, pr_level=s))
                side = r.side(G.n)
                assert r.lam == 2 == oracle.cut_weight(*g, side)
                assert side.sum() == n // 2
