"""Graphs that neither the triangle tests nor the forest packing suit: after a
packing that united little the next waits until half of the vertices are gone.
Exact."""
import numpy as np
import pytest

import graphgen
import oracle

pytestmark = pytest.mark.gpu


def _regular(n, k, wmax, seed):
    rng = np.random.default_rng(seed)
    u = np.concatenate([np.arange(n)] * k)
    v = np.concatenate([rng.permutation(n) for _ in range(k)])
    key = np.unique((np.minimum(u, v) * n + np.maximum(u, v))[u != v])
    return graphgen.from_edges(n, key // n, key % n, rng.integers(1, wmax + 1, len(key)))


def test_poor_packings_are_few(monkeypatch, capfd):
    # random 8-regular graphs, the bound near the mean degree: the packing unites
    # hardly a vertex, the scans a few a round
    import paper_1808_05458_gb300 as mc
    monkeypatch.setenv("MC_VERBOSE", "1")
    for seed in range(4):
        g = _regular(6000, 4, 12, seed)
        with mc.Graph(*g) as G:
            capfd.readouterr()
            r = G.min_cut(mc.options(tail_vertices=-1))
            log = capfd.readouterr().err
        assert r.lam == oracle.noi(*g)[0] == oracle.cut_weight(*g, r.side(6000))
        most, tried = 6000, 0
        for line in log.splitlines():
            if "without scans" in line:
                n, un = (int(line.split(k)[1].split()[0].rstrip(":")) for k in (" n=", "unions="))
                assert n <= most, line
                if un * 8 < n:
                    most = n // 2
                tried += 1
        assert tried > 0
