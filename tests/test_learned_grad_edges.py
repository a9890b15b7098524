"""The proposer's gradient at the edges of the backward kernels' tiles: 64
vertices a tile, eight at a time in the head and the input layer, 32 arcs at a
time in the gather, weights of 1 and above, and a row longer than a tile.

Biases hold every ReLU well on one side of its corner for all vertices, so the
reference (float64, BF16 rounding at the same points) and the kernels take the
same mask, and only sums are left: in FP32 those of at most 200 terms are within
200 * 2^-24 < 2^-16 of exact, so that at most one value in 2^8 may round to the other
BF16 neighbour, a step of 2^-8, at each of ten rounding points: a norm of
10 * 2^-4 * 2^-8 = 2.5e-3.  A vertex left out or counted twice is 1/130 = 7.7e-3
and more.

The smoothed features are what 32 steps of a walk leave after centring, scaled
to 1: where that is below 2^-40 of the start (three vertices: 2^-52), its 64-bit
value is rounding and nothing is compared."""
import numpy as np
import pytest

import oracle
from oracle import gnn
from test_learned_sizes import _hub

pytestmark = pytest.mark.gpu

TOL = 10 * 2.0 ** -12
BLOCKS = [(gnn.P_WIN, gnn.P_BIN), (gnn.P_BIN, gnn.P_W0)]
for _l in range(gnn.L):
    _o = gnn.P_W0 + _l * gnn.P_LAYER
    BLOCKS += [(_o, _o + gnn.K * gnn.H), (_o + gnn.K * gnn.H, _o + gnn.P_LAYER)]
BLOCKS += [(gnn.P_WOUT, gnn.P_BOUT), (gnn.P_BOUT, gnn.P_TOTAL)]


def _params(n):
    """Glorot weights; biases of alternating sign, larger than the sums they are added to."""
    p = gnn.glorot(n).astype(np.float32).astype(np.float64)
    sign = np.where(np.arange(gnn.H) % 2 == 0, 1.0, -1.0)
    p[gnn.P_BIN:gnn.P_BIN + gnn.H] = 4 * sign
    for l, scale in enumerate((16, 64, 256)):
        o = gnn.P_W0 + l * gnn.P_LAYER + gnn.K * gnn.H
        p[o:o + gnn.H] = scale * sign
    p[gnn.P_WOUT:gnn.P_TOTAL] *= 2.0 ** -12
    return p


def _side(n):
    side = np.zeros(n, np.uint8)
    side[np.random.default_rng(n).permutation(n)[:max(1, n // 7)]] = 1
    return side


def _resolved(g):
    n, _, _, _, _, d = G = gnn.features(*g)[1]
    u = lambda h: 2 * (((h >> 40) & 0xFFFFFF) / 2.0 ** 24) - 1
    h = [oracle.splitmix64(gnn.FEAT_SEED ^ oracle.splitmix64(v)) for v in range(n)]
    R = np.array([[u(x), u(oracle.splitmix64(x))] for x in h])
    for _ in range(gnn.SMOOTH):
        R = (R + gnn._aggregate(G, R)) / 2
    left = np.abs(R - (d @ R) / d.sum()).max(0)
    return ((left == 0) | (left > 2.0 ** -40)).all()


def _case(n, wmax):
    g, params, side = _hub(n, wmax), _params(n), _side(n)
    _, (_, _, _, _, zs) = gnn.forward(params, *g, bf16_round=True)
    if not _resolved(g):
        pytest.skip("the walk's remainder is below the resolution of 64 bits")
    assert all(np.abs(z).min() > 2.0 ** -4 * np.abs(z).max() for z in zs)
    return g, params, side


@pytest.mark.parametrize("n,wmax", [(2, 1), (3, 4), (7, 1), (8, 3), (9, 1), (31, 2), (33, 1), (63, 5), (64, 1), (65, 7),
                                    (127, 1), (128, 3), (129, 1), (130, 3)])
def test_gradient_at_tile_edges(n, wmax):
    import paper_1808_05458_gb300 as mc
    g, params, side = _case(n, wmax)
    bits = np.packbits(side, bitorder="little")
    bits = np.concatenate([bits, np.zeros((-len(bits)) % 4, np.uint8)]).view(np.uint32)
    P = mc.Proposer(params.astype(np.float32))
    with mc.Graph(*g) as G:
        loss, grad = P.grad(G, bits)
    P.close()
    ref_loss, ref = gnn.loss_and_grad(params, *g, side.astype(np.int64), bf16_round=True)
    assert abs(loss - ref_loss) < TOL * ref_loss
    for a, b in BLOCKS:
        assert np.linalg.norm(grad[a:b] - ref[a:b]) <= TOL * np.linalg.norm(ref[a:b]), (a, b)
