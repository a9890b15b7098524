"""The bytes a solve reports are those its kernels have to move: on a core that
one packing unites but for a few vertices, the contraction reads the rows outside
that block and no longer every arc, and neither does anything else of the solve."""
import pytest

import graphgen

pytestmark = pytest.mark.gpu


def test_rows_outside_one_block():
    import paper_1808_05458_gb300 as mc
    g = graphgen.rmat_kcore(3, 17, k=10)
    n, arcs = len(g[0]) - 1, len(g[1])
    assert arcs >= 1 << 20
    with mc.Graph(*g) as G:
        st = G.min_cut().stats
    assert st["scan_launches"] == 0 and st["rounds"] <= 2
    # forests: 20 bytes a unit of the bound (below 20) and vertex
    assert 4 * n < st["bytes_alg"] < 20 * 20 * n + 64 * n
    assert st["bytes_alg"] < 8 * arcs
