"""The block-per-graph batched solver against the oracle: sizes around its
limits (the matrix, the shares of shared memory, the most vertices), graphs it
leaves to the warp-per-graph solver (rows not canonical, heavy weights, an
empty row, one vertex too many), and input that must be refused.  Whole
numbers: lambda and the weight of the side are compared exactly."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mc():
    import paper_1808_05458_gb300 as m
    m.load_library()
    return m


def _csr(n, u, v, w):
    """Canonical rows of the edges, parallel ones merged."""
    key = np.concatenate([u, v]).astype(np.int64) * n + np.concatenate([v, u])
    k, inv = np.unique(key, return_inverse=True)
    ww = np.bincount(inv, weights=np.concatenate([w, w])).astype(np.int32)
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(k // n, minlength=n))
    return rp, (k % n).astype(np.int32), ww


def _random(n, deg, wmax, seed):
    rng = np.random.default_rng(seed)
    tree = np.array([rng.integers(0, v) for v in range(1, n)], dtype=np.int64)
    extra = max(int(n * deg / 2) - (n - 1), 0)
    a, b = rng.integers(0, n, extra), rng.integers(0, n, extra)
    keep = a != b
    u = np.concatenate([np.arange(1, n), a[keep]])
    v = np.concatenate([tree, b[keep]])
    p = rng.permutation(n)
    return _csr(n, p[u], p[v], rng.integers(1, wmax + 1, len(u)))


def _complete(n, wmax, seed):
    u, v = np.triu_indices(n, 1)
    return _csr(n, u, v, np.random.default_rng(seed).integers(1, wmax + 1, len(u)))


def _two_cliques(k, w, cross):
    u, v = np.triu_indices(k, 1)
    c = np.arange(cross)
    return _csr(2 * k, np.concatenate([u, u + k, c]), np.concatenate([v, v + k, c + k]),
                np.concatenate([np.full(2 * len(u), w), np.ones(cross, int)]))


def _run(mc, gs):
    rp = np.concatenate([g[0] for g in gs])
    vo = np.concatenate([[0], np.cumsum([len(g[0]) - 1 for g in gs])])
    ao = np.concatenate([[0], np.cumsum([len(g[1]) for g in gs])])
    lam, bw, bo, _ = mc.batch_min_cut(rp, np.concatenate([g[1] for g in gs]), np.concatenate([g[2] for g in gs]),
                                      vo, ao, bitmaps=True)
    return lam, [mc.bitmap_to_side(bw[bo[k]:bo[k + 1]], len(gs[k][0]) - 1) for k in range(len(gs))]


def _check(mc, gs):
    lam, sides = _run(mc, gs)
    for g, l, side in zip(gs, lam, sides):
        n = len(g[0]) - 1
        assert l == oracle.noi(*g)[0]
        assert side[0] == 0 and 0 < side.sum() < n
        assert oracle.cut_weight(*g, side) == l


@pytest.mark.parametrize("wmax", [1, 100, 0x7fff])
def test_sizes_around_the_limits(mc, wmax):
    sizes = [2, 3, 31, 32, 33, 63, 64, 65, 130, 225, 511, 512, 513, 1025, 2047, 2048, 2049]
    _check(mc, [_random(n, d, wmax, 7 * n + int(d)) for n in sizes for d in (2.0, 5.0, 16.0)])


def test_shapes_of_graphs(mc):
    star = _csr(700, np.zeros(699, int), np.arange(1, 700), np.arange(1, 700))
    path = _csr(2048, np.arange(2047), np.arange(1, 2048), np.full(2047, 5))
    cycle = _csr(1000, np.arange(1000), (np.arange(1000) + 1) % 1000, np.full(1000, 3))
    _check(mc, [star, path, cycle, _complete(64, 9, 1), _complete(66, 1, 2), _complete(200, 50, 3),
                _complete(255, 1, 4), _complete(257, 1, 5), _two_cliques(40, 3, 7), _two_cliques(120, 1, 20)])


def test_many_small_graphs(mc):
    # more than half of the batch between the matrix's and the warps' sizes
    _check(mc, [_random(n, 6.0, 100, 31 * n + k) for k in range(14) for n in range(33, 96)]
           + [_random(n, 6.0, 100, n) for n in (20, 96, 700)])


def test_left_to_the_warps(mc):
    # rows with parallel and unsorted arcs, weights above 15 bits, an isolated
    # vertex, two components, among graphs that stay
    loose = [graphgen.random_connected(n, 4 * n, seed=n, wmax=20) for n in (40, 300, 900)]
    heavy = _random(300, 6.0, 100, 5)
    heavy = (heavy[0], heavy[1], (heavy[2] * 4000).astype(np.int32))
    u = np.arange(1, 99)
    lone = _csr(100, u, u - 1, np.full(98, 2))
    a = np.arange(1, 60)
    apart = _csr(120, np.concatenate([a, a + 60]), np.concatenate([a - 1, a + 59]), np.full(118, 2))
    _check(mc, [_random(500, 8.0, 9, 1)] + loose + [heavy, lone, apart, _random(80, 8.0, 9, 2)])


@pytest.mark.parametrize("fault", ["range", "mirror", "weight", "negative", "offsets"])
def test_faulty_graphs_are_refused(mc, fault):
    good = _random(400, 8.0, 9, 3)
    rp, col, w = (x.copy() for x in _random(400, 8.0, 9, 4))
    if fault == "range":
        col[rp[200] - 1] = 400
    elif fault == "mirror":
        u = next(v for v in range(10, 400) if col[rp[v + 1] - 1] < 399)
        col[rp[u + 1] - 1] = 399
    elif fault == "weight":
        w[7] += 1
    elif fault == "negative":
        w[7] = -1
    else:
        rp[100] = rp[101] + 1
    with pytest.raises(Exception):
        _run(mc, [good, (rp, col, w), good])
    _check(mc, [good])


@pytest.mark.parametrize("wmax", [1, 3])
def test_dense_rows_of_small_weights(mc, wmax):
    # mean degrees far above the bound: units stay at the weights' size
    _check(mc, [_random(n, d, wmax, 13 * n + int(d)) for n in (120, 400) for d in (40.0, 60.0)]
           + [_two_cliques(60, 1, 5), _complete(150, wmax, 6)])


def test_large_batch_in_chunks(mc):
    # more arcs than a batch that is copied whole; graphs for the warps among
    # them, and a fault in the last chunk
    kinds = [_random(n, d, 50, 17 * n) for n, d in ((1500, 6.0), (2000, 5.0), (50, 8.0), (700, 12.0), (2100, 4.0))]
    kinds.append(graphgen.random_connected(300, 1500, seed=3, wmax=9))
    want = [oracle.noi(*g)[0] for g in kinds]
    order = np.random.default_rng(1).integers(0, len(kinds), 6000)
    gs = [kinds[k] for k in order]
    assert sum(len(g[1]) for g in gs) >= 32 << 20
    for _ in range(2):
        lam, sides = _run(mc, gs)
        assert lam.tolist() == [want[k] for k in order]
        for j in range(0, len(gs), 241):
            assert oracle.cut_weight(*gs[j], sides[j]) == lam[j]
    rp, col, w = (x.copy() for x in kinds[0])
    w[5] += 1
    with pytest.raises(Exception):
        _run(mc, gs + [(rp, col, w)])
    assert _run(mc, gs)[0].tolist() == [want[k] for k in order]
