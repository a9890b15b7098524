"""Graphs numbered along a path: the parents of the certificates' first unions
then hang in chains as long as the graph, and every walk has to shorten them.
Lambda in closed form, and a solve no dearer than that of the same graph with
shuffled numbers by more than 4 ms: a walk over a quarter of the 2^20 vertices
takes 2^18 loads that wait for one another, 20 ns each at the very least."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N = 1 << 20


def _edges(kind):
    i = np.arange(N - 1)
    if kind == "band":
        u = np.repeat(np.arange(N), 4)
        v = u + np.tile(np.arange(1, 5), N)
        return u[v < N], v[v < N], np.ones(int((v < N).sum()), int), 4
    if kind == "cycle":
        return np.arange(N), (np.arange(N) + 1) % N, np.full(N, 3), 6
    w = {"path": np.full(N - 1, 2), "rising": i + 1, "falling": N - 1 - i}[kind]
    return i, i + 1, w, int(w.min())


def _csr(u, v, w):
    key = np.concatenate([u, v]).astype(np.int64) * N + np.concatenate([v, u])
    o = np.argsort(key, kind="stable")
    rp = np.zeros(N + 1, np.int32)
    rp[1:] = np.cumsum(np.bincount(key // N, minlength=N))
    return rp, (key[o] % N).astype(np.int32), np.concatenate([w, w])[o].astype(np.int32)


def _weight(u, v, w, side):
    return int(w[side[u] != side[v]].sum())


@pytest.mark.parametrize("kind", ["path", "rising", "falling", "cycle", "band"])
@pytest.mark.parametrize("opt", [{}, {"pr_level": 0}, {"tail_vertices": -1}])
def test_numbered_along_a_path(kind, opt):
    import paper_1808_05458_gb300 as mc
    if kind == "cycle" and opt.get("pr_level") == 0:
        return  # a scan of a cycle unites one edge
    u, v, w, lam = _edges(kind)
    p = np.random.default_rng(1).permutation(N)
    ms = []
    for a, b in ((u, v), (p[u], p[v])):
        with mc.Graph(*_csr(a, b, w)) as G:
            best = np.inf
            for _ in range(3):
                r = G.min_cut(mc.options(**opt))
                best = min(best, r.stats["ms_total"])
            side = r.side(N)
        assert r.lam == lam == _weight(a, b, w, side)
        assert side[0] == 0 and 0 < side.sum() < N
        ms.append(best)
    assert ms[0] < ms[1] + 4.0, ms
