"""A contraction that leaves few blocks goes on to the dense rounds without a
graph in between: cliques (which unite) joined at random, as many as the matrix
holds and one more or less, with weights from 1 to beyond what the matrix's sums
or keys hold (those build the graph as ever).  Exact against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _cliques(k, size, inner, cross_w, per, seed):
    rng = np.random.default_rng(seed)
    a, b = np.triu_indices(size, 1)
    u = (np.arange(k)[:, None] * size + a).ravel()
    v = (np.arange(k)[:, None] * size + b).ravel()
    w = np.full(len(u), inner)
    # a ring keeps it connected; random links besides
    cu = np.concatenate([np.arange(k - 1), rng.integers(0, k, per * k)])
    cv = np.concatenate([np.arange(1, k), rng.integers(0, k, per * k)])
    keep = cu != cv
    cu, cv = cu[keep], cv[keep]
    u = np.concatenate([u, cu * size + rng.integers(0, size, len(cu))])
    v = np.concatenate([v, cv * size + rng.integers(0, size, len(cv))])
    w = np.concatenate([w, rng.integers(1, cross_w + 1, len(cu))])
    n = k * size
    key = np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u])
    uniq, inv = np.unique(key, return_inverse=True)
    ww = np.bincount(inv, weights=np.concatenate([w, w])).astype(np.int32)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(uniq // n, minlength=n))
    return rp, (uniq % n).astype(np.int32), ww


@pytest.mark.parametrize("k", [1, 2, 3, 32, 33, 223, 224, 225])
@pytest.mark.parametrize("inner,cross", [(40, 9), (1, 1), (3000, 700), (1 << 19, 1 << 17), (1 << 21, 1 << 20)])
def test_blocks_around_the_matrix(k, inner, cross):
    import paper_1808_05458_gb300 as mc
    size = max(12, -(-300 // k))
    g = _cliques(k, size, inner, cross, 3, 97 * k + cross)
    with mc.Graph(*g) as G:
        for o in (mc.options(), mc.options(seed=5, pr_level=1), mc.options(bound=mc.MC_BOUND_LP)):
            r = G.min_cut(o)
            side = r.side(G.n)
            assert r.lam == oracle.noi(*g)[0]
            assert side[0] == 0 and 0 < side.sum() < G.n and oracle.cut_weight(*g, side) == r.lam
