"""The proposer's forward kernels at the edges of their tiles: vertices around
the 64-row tiles and the groups of eight of the head, rows around the 128 arcs
from which a whole warp takes a walk's row, weights of 1 and above.  Logits and
loss against float64 (oracle/gnn.py) with BF16 rounding at the same points.  A
value rounded to BF16 on either side may take the other side of a tie, a step of
2^-8 relative at each of the six rounding points between input and output:
6 * 2^-8 = 2.4e-2."""
import numpy as np
import pytest

import graphgen
from oracle import gnn

pytestmark = pytest.mark.gpu

TOL = 6 * 2.0 ** -8


def _hub(n, wmax):
    """A connected graph with vertex 0 next to all others."""
    rng = np.random.default_rng(n)
    e = {(0, v): 1 for v in range(1, n)}
    for _ in range(3 * n):
        a, b = sorted(int(x) for x in rng.integers(0, n, 2))
        if a != b:
            e[(a, b)] = 1
    u = np.array([k[0] for k in e])
    v = np.array([k[1] for k in e])
    w = rng.integers(1, wmax + 1, len(u))
    s, d, ww = np.concatenate([u, v]), np.concatenate([v, u]), np.concatenate([w, w])
    o = np.lexsort((d, s))
    rp = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(s, minlength=n), out=rp[1:])
    return rp.astype(np.int32), d[o].astype(np.int32), ww[o].astype(np.int32)


@pytest.mark.parametrize("n,wmax", [(9, 1), (63, 5), (64, 1), (65, 7), (129, 1), (130, 3), (321, 1)])
def test_forward_at_tile_edges(n, wmax):
    import paper_1808_05458_gb300 as mc
    g = _hub(n, wmax)
    params = gnn.glorot(n)
    side = (np.random.default_rng(n).random(n) < 0.4).astype(np.uint8)
    bits = np.packbits(side, bitorder="little")
    bits = np.concatenate([bits, np.zeros((-len(bits)) % 4, np.uint8)]).view(np.uint32)
    P = mc.Proposer(params.astype(np.float32))
    with mc.Graph(*g) as G:
        logits = P.forward(G)
        loss, _ = P.grad(G, bits)
    P.close()
    ref_s, _ = gnn.forward(params, *g, bf16_round=True)
    ref_loss, _ = gnn.loss_and_grad(params, *g, side.astype(np.int64), bf16_round=True)

    def rel(a, b):
        return np.linalg.norm(np.asarray(a, np.float64) - b) / max(np.linalg.norm(b), 1e-30)

    assert rel(logits, ref_s) < TOL
    assert abs(loss - ref_loss) < TOL * abs(ref_loss)
