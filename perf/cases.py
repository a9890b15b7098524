"""Workloads of the exact minimum-cut library, as a user's program runs them.

Every case goes through the package's public entry points: one graph resident on the GPU and
solved (``Graph.min_cut``), one graph handed over as host arrays and solved (graph creation,
solve, release), many small graphs at once (``batch_min_cut``), and the learned proposer's
training pass (``Proposer.grad``).  The graphs are the families this repository's configurations,
tests and benchmark name -- threshold random hyperbolic graphs (exponent 5), planted cuts, k-cores
of R-MAT graphs, batches of random connected graphs -- drawn on the GPU from the seed alone.
"""
import math

import numpy as np
import torch

import paper_1808_05458_gb300 as mc

DEV = "cuda"


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest call: one weighted graph of a few hundred vertices, handed over as host
        # arrays and thrown away again (a serving process that gets one graph per request)
        dict(name="oneshot_random_200", family="random", n=200, deg=12.0, wmax=100, input="host"),
        # the small plain workload: two random blocks joined by a few edges, lambda below delta,
        # on expander-like blocks where no local region certifies anything
        dict(name="planted_2x2048_d24", family="planted", n=2048, deg=24.0, cross=8, input="device",
             bound="degree", approx=0),
        # an ordinary graph of odd size, where launches and round trips are most of a solve
        dict(name="rhg_30011_d24", family="rhg", n=30011, deg=24.0, input="device", bound="degree", approx=0),
        # the benchmark's graph: the paper's synthetic family at 2^20 points, resident on the device
        dict(name="rhg_2e20_d32", family="rhg", n=1 << 20, deg=32.0, input="device", bound="degree", approx=0),
        # the same, end to end: page-locked host arrays of an unweighted graph in, lambda and the
        # side back in host memory, nothing kept
        dict(name="oneshot_rhg_2e20_d32", family="rhg", n=1 << 20, deg=32.0, input="host", bound="degree",
             approx=0),
        # the large end of the family: 134 M edges, rows twice as long, a higher bound
        dict(name="rhg_2e22_d64", family="rhg", n=1 << 22, deg=64.0, input="device", bound="degree", approx=0),
        # the paper's real-world shape: a weighted, skewed k-core with hubs of 10^4..10^5 arcs
        dict(name="rmat_s20_k10", family="rmat", scale=20, k=10, wmax=4, input="device", bound="degree", approx=0),
        # a deep k-core of the same: few vertices, long rows around hubs, a bound near 100
        dict(name="rmat_s18_k50", family="rmat", scale=18, k=50, wmax=4, input="device", bound="degree", approx=0),
        # a minimum cut below the minimum degree found with the label-propagation bound (VieCut)
        dict(name="planted_rhg_2x2e18_d64_lp", family="planted_rhg", n=1 << 18, deg=64.0, cross=8,
             input="device", bound="lp", approx=0),
        # many small weighted graphs in one call, from page-locked host arrays, with their sides
        dict(name="batch_4096_n50_2000", family="batch", graphs=4096, nmin=50, nmax=2000, dmin=4.0, dmax=16.0,
             wmax=100, sides=True),
        # a small batch of small graphs: far fewer graphs than the GPU has warps
        dict(name="batch_96_n50_400", family="batch", graphs=96, nmin=50, nmax=400, dmin=4.0, dmax=16.0,
             wmax=100, sides=False),
        # one training pass of the learned proposer (loss and gradient) on a planted-cut graph
        dict(name="proposer_grad_2x2e14_d32", family="proposer", n=1 << 14, deg=32.0, cross=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["random", "planted", "rhg", "rhg", "rhg", "rmat", "rmat", "planted_rhg", "batch", "batch",
                       "proposer"])
    if kind == "random":
        return dict(family=kind, n=_log_int(rng, 30, 2000), deg=round(rng.uniform(6, 20), 1),
                    wmax=rng.choice([3, 10, 100]), input="host")
    if kind == "planted":
        return dict(family=kind, n=_log_int(rng, 300, 4000), deg=round(rng.uniform(20, 40), 1),
                    cross=rng.randint(2, 8), input="device", bound="degree", approx=0)
    if kind == "rhg":
        deg = rng.choice([16.0, 24.0, 32.0, 48.0, 64.0])
        return dict(family=kind, n=_log_int(rng, 3000, 1 << 22), deg=deg,
                    input=rng.choice(["device", "device", "host"]), bound=rng.choice(["degree", "degree", "lp"]),
                    approx=rng.choice([0, 0, 0, 500]))
    if kind == "rmat":
        return dict(family=kind, scale=rng.randint(16, 20), k=rng.randint(10, 50), wmax=rng.choice([1, 4, 4]),
                    input="device", bound="degree", approx=0)
    if kind == "planted_rhg":
        return dict(family=kind, n=_log_int(rng, 1 << 13, 1 << 19), deg=rng.choice([48.0, 64.0]),
                    cross=rng.randint(2, 8), input="device", bound=rng.choice(["degree", "lp"]), approx=0)
    if kind == "batch":
        return dict(family=kind, graphs=_log_int(rng, 16, 4096), nmin=50, nmax=rng.randint(200, 2000), dmin=4.0,
                    dmax=16.0, wmax=rng.choice([4, 100]), sides=False)
    return dict(family=kind, n=_log_int(rng, 1 << 11, 1 << 16), deg=rng.choice([24.0, 32.0, 48.0]),
                cross=rng.randint(2, 8))


# ------------------------------------------------------------- graphs (torch)
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed & (2**62 - 1))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _components(n, u, v):
    """The smallest vertex of every vertex's component."""
    lab = torch.arange(n, device=DEV)
    while True:
        a, b = lab[u], lab[v]
        new = lab.clone()
        new.scatter_reduce_(0, a, b, "amin")
        new.scatter_reduce_(0, b, a, "amin")
        while True:
            hop = new[new]
            if torch.equal(hop, new):
                break
            new = hop
        if torch.equal(new, lab):
            return lab
        lab = new


def _largest_component(n, u, v, w):
    """The largest component, its vertices renumbered in order."""
    lab = _components(n, u, v)
    size = torch.bincount(lab, minlength=n)
    keep = lab == torch.argmax(size)
    if bool(keep.all()):
        return n, u, v, w
    new = torch.cumsum(keep, 0) - 1
    ok = keep[u]
    return int(keep.sum()), new[u[ok]], new[v[ok]], None if w is None else w[ok]


def _csr(n, u, v, w):
    """(row_ptr, col, w) as int32 from distinct undirected edges; rows sorted, w None: unweighted."""
    key = torch.cat([u * n + v, v * n + u])
    if w is None:
        key = torch.sort(key)[0]
        ww = None
    else:
        key, at = torch.sort(key)
        ww = torch.cat([w, w])[at].to(torch.int32)
    src = key // n
    rp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(torch.bincount(src, minlength=n), 0)
    return rp.to(torch.int32), (key - src * n).to(torch.int32), ww


def _hyperbolic_pairs(th, r, R, width=0.5, bands=16, most=1 << 26):
    """The edges of a threshold hyperbolic graph: pairs of points at distance <= R.  Points go in
    radial bands, outermost first; a point looks for neighbours in its own and the inner bands."""
    band = torch.clamp(((R - r) / width).to(torch.int64), max=bands - 1)
    order = torch.argsort(band.to(torch.float64) * 8.0 + th)
    th, r, band = th[order], r[order], band[order]
    ch, sh = torch.cosh(r), torch.sinh(r)
    start = [0] + torch.cumsum(torch.bincount(band, minlength=bands), 0).tolist()
    two_pi = 2 * math.pi
    us, vs = [], []
    for b in range(bands):
        lo, hi = start[b], start[b + 1]
        if hi == lo:
            continue
        inner = 0.0 if b == bands - 1 else max(0.0, R - width * (b + 1))
        if inner > 0:
            c = (ch[:hi] * math.cosh(inner) - math.cosh(R)) / (sh[:hi] * math.sinh(inner)).clamp_min(1e-300)
            d = torch.acos(torch.clamp(c, -1.0, 1.0)) + 1e-9
        else:
            d = torch.full((hi,), math.pi, dtype=torch.float64, device=DEV)
        m = hi - lo
        ring = torch.cat([th[lo:hi] - two_pi, th[lo:hi], th[lo:hi] + two_pi])
        a = torch.searchsorted(ring, th[:hi] - d)
        cnt = torch.minimum(torch.searchsorted(ring, th[:hi] + d, right=True) - a, torch.tensor(m, device=DEV))
        upto = torch.cumsum(cnt, 0)
        i0 = 0
        while i0 < hi:
            base = int(upto[i0 - 1]) if i0 else 0
            i1 = min(hi, max(i0 + 1, int(torch.searchsorted(upto, torch.tensor(base + most, device=DEV)))))
            k = cnt[i0:i1]
            i = torch.repeat_interleave(torch.arange(i0, i1, device=DEV), k)
            first = torch.cumsum(k, 0) - k
            j = lo + (a[i] + torch.arange(i.numel(), device=DEV) - first[i - i0]) % m
            ok = (j > i) & (ch[i] * ch[j] - sh[i] * sh[j] * torch.cos(th[i] - th[j]) <= math.cosh(R))
            us.append(i[ok])
            vs.append(j[ok])
            i0 = i1
    return order[torch.cat(us)], order[torch.cat(vs)]


def _hyperbolic(g, n, deg):
    """A random hyperbolic graph of exponent 5 and about this average degree: (n, u, v) of its
    largest component, vertices in sampling order."""
    alpha = 2.0
    U, th = _rand(g, n), _rand(g, n) * 2 * math.pi

    def radii(R, x):
        return torch.acosh(1 + x * (math.cosh(alpha * R) - 1)) / alpha

    R = 2 * math.log(2 / math.pi * (alpha / (alpha - 0.5)) ** 2 * n / deg)
    # the asymptotic radius gives too few or too many edges at small sizes: corrected on a
    # thinned ring of the same density
    k = min(n, 1 << 15)
    Rk = R + 2 * math.log(k / n)
    for _ in range(2):
        u, _v = _hyperbolic_pairs(th[:k], radii(Rk, U[:k]), Rk)
        Rk += 2 * math.log(max(1, 2 * u.numel()) / k / deg)
    R = Rk + 2 * math.log(n / k)
    u, v = _hyperbolic_pairs(th, radii(R, U), R)
    n, u, v, _ = _largest_component(n, u, v, None)
    return n, u, v


def _joined(g, a, b, cross):
    """Two graphs and `cross` distinct random edges between them, vertices in random order: (n, u, v, the
    vertices of the second)."""
    (na, ua, va), (nb, ub, vb) = a, b
    x = torch.unique((_rand(g, 8 * cross) * na).to(torch.int64) * nb + (_rand(g, 8 * cross) * nb).to(torch.int64))
    x = x[torch.argsort(_rand(g, x.numel()))][:cross]
    perm = torch.argsort(_rand(g, na + nb))
    u, v = torch.cat([ua, na + ub, x // nb]), torch.cat([va, na + vb, na + x % nb])
    return na + nb, perm[u], perm[v], perm[na:]


def _block(g, n, deg):
    """A uniform random graph with about n * deg / 2 distinct edges (largest component)."""
    m = int(n * deg / 2)
    u, v = (_rand(g, m) * n).to(torch.int64), (_rand(g, m) * n).to(torch.int64)
    key = torch.unique(torch.minimum(u, v)[u != v] * n + torch.maximum(u, v)[u != v])
    return _largest_component(n, key // n, key % n, None)[:3]


def _rmat_core(g, scale, k, wmax, edge_factor=16, a=0.57, b=0.19, c=0.19):
    """The k-core of an R-MAT graph (symmetrised, no loops or repeats), its largest component;
    weights uniform in 1..wmax."""
    n, m = 1 << scale, edge_factor << scale
    u = torch.zeros(m, dtype=torch.int64, device=DEV)
    v = torch.zeros(m, dtype=torch.int64, device=DEV)
    for _ in range(scale):
        r = torch.rand(m, generator=g, device=DEV)
        u = 2 * u + (r >= a + b)
        v = 2 * v + (((r >= a) & (r < a + b)) | (r >= a + b + c))
    key = torch.unique(torch.minimum(u, v)[u != v] * n + torch.maximum(u, v)[u != v])
    u, v = key // n, key % n
    while True:
        deg = torch.bincount(u, minlength=n) + torch.bincount(v, minlength=n)
        ok = (deg[u] >= k) & (deg[v] >= k)
        if bool(ok.all()):
            break
        u, v = u[ok], v[ok]
    alive = deg > 0
    new = torch.cumsum(alive, 0) - 1
    w = None if wmax == 1 else torch.randint(1, wmax + 1, u.shape, generator=g, device=DEV)
    return _largest_component(int(alive.sum()), new[u], new[v], w)


def _batch(g, graphs, nmin, nmax, dmin, dmax, wmax):
    """Random connected weighted graphs (a random spanning tree and uniform extra edges each),
    concatenated: (row_ptr, col, w, vtx_off, arc_off) on the host as batch_min_cut takes them."""
    n = torch.linspace(nmin, nmax, graphs, device=DEV).round().to(torch.int64)  # sizes evenly spread
    n = n[torch.argsort(_rand(g, graphs))]
    d = dmin + (dmax - dmin) * _rand(g, graphs)
    voff = torch.zeros(graphs + 1, dtype=torch.int64, device=DEV)
    voff[1:] = torch.cumsum(n, 0)
    V = int(voff[-1])
    gid = torch.repeat_interleave(torch.arange(graphs, device=DEV), n)
    at = torch.arange(V, device=DEV) - voff[gid]
    perm = torch.argsort(gid.to(torch.float64) + _rand(g, V))
    child = at > 0
    up = (_rand(g, V) * at).to(torch.int64)
    extra = torch.clamp((n * d / 2).round().to(torch.int64) - (n - 1), min=0)
    eg = torch.repeat_interleave(torch.arange(graphs, device=DEV), extra)
    xu = voff[eg] + (_rand(g, eg.numel()) * n[eg]).to(torch.int64)
    xv = voff[eg] + (_rand(g, eg.numel()) * n[eg]).to(torch.int64)
    u = torch.cat([perm[child], xu])
    v = torch.cat([perm[(voff[gid] + up)[child]], xv])
    key = torch.unique(torch.minimum(u, v)[u != v] * V + torch.maximum(u, v)[u != v])
    u, v = key // V, key % V
    w = torch.randint(1, wmax + 1, u.shape, generator=g, device=DEV)
    rp, col, w = _csr(V, u, v, w)
    aoff = rp[voff].to(torch.int64)
    # each graph's own offsets (n + 1 of them) and local vertex ids
    slot = torch.arange(V, device=DEV) + gid
    local = torch.empty(V + graphs, dtype=torch.int32, device=DEV)
    local[slot] = (rp[:-1].to(torch.int64) - aoff[gid]).to(torch.int32)
    local[voff[1:] + torch.arange(graphs, device=DEV)] = (aoff[1:] - aoff[:-1]).to(torch.int32)
    row = torch.repeat_interleave(gid, (rp[1:] - rp[:-1]).to(torch.int64))
    col = (col.to(torch.int64) - voff[row]).to(torch.int32)
    return local, col, w, voff, aoff


def _graph(case, seed):
    """(row_ptr, col, w or None) on the GPU; a planted cut's graph with the vertices of one side."""
    g = _gen(seed)
    kind = case["family"]
    if kind == "rhg":
        return (*_csr(*_hyperbolic(g, case["n"], case["deg"]), None), None)
    if kind in ("planted_rhg", "proposer"):
        a, b = (_hyperbolic(g, case["n"], case["deg"]) for _ in range(2))
        n, u, v, second = _joined(g, a, b, case["cross"])
        return (*_csr(n, u, v, None), second)
    if kind == "planted":
        a, b = (_block(g, case["n"], case["deg"]) for _ in range(2))
        n, u, v, second = _joined(g, a, b, case["cross"])
        return (*_csr(n, u, v, None), second)
    if kind == "rmat":
        return (*_csr(*_rmat_core(g, case["scale"], case["k"], case["wmax"])), None)
    if kind == "random":
        rp, col, w, _, _ = _batch(g, 1, case["n"], case["n"], case["deg"], case["deg"], case["wmax"])
        return rp, col, w, None
    raise ValueError(kind)


def _pinned(t):
    return t.cpu().pin_memory().numpy()


def _proposer_params(seed):
    """Glorot-uniform weights, small biases: the network's 25409 parameters."""
    rng = np.random.default_rng(seed)

    def layer(fan_in, fan_out):
        a = math.sqrt(6.0 / (fan_in + fan_out))
        return [rng.uniform(-a, a, fan_in * fan_out), rng.uniform(-0.05, 0.05, fan_out)]

    parts = layer(8, 64) + layer(128, 64) + layer(128, 64) + layer(128, 64) + layer(64, 1)
    return np.concatenate(parts).astype(np.float32)


def _most_vertices(case):
    if case["family"] == "rmat":
        return 1 << case["scale"]
    return case["n"] * (2 if case["family"] in ("planted", "planted_rhg", "proposer") else 1)


# ------------------------------------------------------------------- protocol
def prepare(case, seed):
    if case["family"] == "batch":
        arrays = _batch(_gen(seed), case["graphs"], case["nmin"], case["nmax"], case["dmin"], case["dmax"],
                        case["wmax"])
        return dict(kind="batch", arrays=[_pinned(t) for t in arrays], sides=case["sides"])
    rp, col, w, second = _graph(case, seed)
    if case["family"] == "proposer":
        # labels: one side of the planted cut (the second block's vertices)
        n = rp.numel() - 1
        side = np.zeros(n + (-n) % 32, dtype=np.uint8)
        side[second.cpu().numpy()] = 1
        bits = np.packbits(side, bitorder="little").view(np.uint32)
        return dict(kind="proposer", graph=mc.Graph(rp, col, w), net=mc.Proposer(_proposer_params(seed)), bits=bits)
    opts = mc.options(bound=mc.MC_BOUND_LP if case.get("bound") == "lp" else mc.MC_BOUND_DEGREE,
                      approx_milli=case.get("approx", 0))
    # the caller's buffer for the side's bitmap, large enough for any graph of the case
    words = (_most_vertices(case) + 31) // 32
    if case["input"] == "host":
        return dict(kind="host", arrays=[_pinned(t) for t in (rp, col, w) if t is not None], opts=opts,
                    side=np.zeros(words, dtype=np.uint32))
    return dict(kind="device", graph=mc.Graph(rp, col, w), opts=opts,
                side=torch.zeros(words, dtype=torch.int32, device=DEV))


def run(state):
    if state["kind"] == "device":
        r = state["graph"].min_cut(state["opts"], bitmap_out=state["side"])
        return r.lam, r.bitmap
    if state["kind"] == "host":
        with mc.Graph(*state["arrays"]) as g:
            r = g.min_cut(state["opts"], bitmap_out=state["side"])
        return r.lam, r.bitmap.view(np.int32)
    if state["kind"] == "batch":
        lam, bits, _, _ = mc.batch_min_cut(*state["arrays"], bitmaps=state["sides"])
        return (lam, bits.view(np.int32)) if state["sides"] else lam
    loss, grad = state["net"].grad(state["graph"], state["bits"])
    return {"loss": loss, "grad": grad}


def work(case):
    """The graph read once (offsets, neighbours, and weights where it has any) and the result written once."""
    kind = case["family"]
    if kind == "batch":
        n = case["graphs"] * (case["nmin"] + case["nmax"]) / 2
        arcs = n * (case["dmin"] + case["dmax"]) / 2
        return dict(bytes=4 * n + 8 * arcs + case["graphs"] * 24 + (n / 8 if case["sides"] else 0), flops=2 * arcs)
    weighted = kind == "random" or (kind == "rmat" and case["wmax"] > 1)
    if kind == "rmat":
        # share of the 16 * 2^scale sampled edges, and of the vertices, left in the k-core
        # (measured at scales 16 to 20)
        edges = (16 << case["scale"]) * (0.86 + 0.02 * (case["scale"] - 20) - 0.0065 * (case["k"] - 10))
        n, arcs = (1 << case["scale"]) * 0.24 * (10 / case["k"]) ** 0.75, 2 * edges
    else:
        blocks = 2 if kind in ("planted", "planted_rhg", "proposer") else 1
        n = blocks * case["n"]
        arcs = n * case["deg"]
    if kind == "proposer":
        # three layers forward and backward: the aggregation gathers 64 features along every arc,
        # the dense transforms are n x 128 x 64 (one product forward, two backward); 32 smoothing
        # steps of two features
        return dict(bytes=4 * n + 4 * arcs + 2 * 4 * 25409 + n / 8,
                    flops=3 * (2 * 2 * 64 * arcs + 3 * 2 * 128 * 64 * n) + 32 * 4 * arcs)
    return dict(bytes=4 * n + (8 if weighted else 4) * arcs + n / 8, flops=2 * arcs)


# ------------------------------------------------------------------ 64-bit truth
def _stoer_wagner(n, rp, col, w):
    """lambda by maximum-adjacency phases on a dense matrix."""
    A = np.zeros((n, n), dtype=np.int64)
    np.add.at(A, (np.repeat(np.arange(n), np.diff(rp)), col), w)
    np.fill_diagonal(A, 0)
    best, alive = None, list(range(n))
    while len(alive) > 1:
        B = A[np.ix_(alive, alive)]
        key, done = B[0].copy(), np.zeros(len(alive), dtype=bool)
        done[0] = True
        s = t = 0
        for _ in range(len(alive) - 1):
            s, t = t, int(np.argmax(np.where(done, -1, key)))
            cut = int(key[t])
            done[t] = True
            key += B[t]
        best = cut if best is None else min(best, cut)
        a, b = alive[s], alive[t]
        A[a] += A[b]
        A[:, a] += A[:, b]
        A[a, a] = 0
        alive.pop(t)
    return best


def _splitmix64(x):
    x = x + np.uint64(0x9E3779B97F4A7C15)
    x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return x ^ (x >> np.uint64(31))


def _proposer_grad64(rp, col, params, label):
    """Loss and gradient of the proposer's network on an unweighted graph, in 64 bits."""
    n = rp.numel() - 1
    rp, col = rp.to(torch.int64), col.to(torch.int64)
    src = torch.repeat_interleave(torch.arange(n, device=DEV), rp[1:] - rp[:-1])
    d = (rp[1:] - rp[:-1]).to(torch.float64)

    def mean(h):
        return torch.zeros_like(h).index_add(0, src, h[col]) / d[:, None]

    least = torch.full((n,), math.inf, dtype=torch.float64, device=DEV).scatter_reduce(0, src, d[col], "amin")
    h = _splitmix64(np.uint64(0x51ED270B27A4BB1D) ^ _splitmix64(np.arange(n, dtype=np.uint64)))
    q = np.stack([((x >> np.uint64(40)) & np.uint64(0xFFFFFF)).astype(np.float64) / 2.0**23 - 1
                  for x in (h, _splitmix64(h))], axis=1)
    q = torch.from_numpy(q).to(DEV)
    for _ in range(32):
        q = (q + mean(q)) / 2
    q = q - (d @ q) / d.sum()
    q = q / q.abs().amax(0)
    x = torch.stack([torch.ones_like(d), torch.log1p(d) / 8, torch.log1p(d) / 8,
                     torch.clamp(d / d.min() - 1, max=8.0) / 8, torch.log1p(mean(d[:, None])[:, 0]) / 8,
                     torch.log1p(least) / 8, q[:, 0], q[:, 1]], dim=1)
    p = torch.from_numpy(params).to(DEV).to(torch.float64).requires_grad_()
    h = torch.relu(x @ p[:512].view(8, 64) + p[512:576])
    at = 576
    for _ in range(3):
        W, b = p[at:at + 8192].view(128, 64), p[at + 8192:at + 8256]
        h = torch.relu(torch.cat([h, mean(h)], dim=1) @ W + b)
        at += 8256
    s = h @ p[at:at + 64] + p[at + 64]
    y = torch.from_numpy(label).to(DEV).to(torch.float64)
    bce = torch.nn.functional.binary_cross_entropy_with_logits
    loss = torch.minimum(bce(s, y), bce(s, 1 - y))
    loss.backward()
    return float(loss.detach()), p.grad.cpu().numpy()


def exact(case, seed):
    """The smallest graphs' lambda (a minimum cut's side has no single answer) and the proposer's loss and
    gradient; the other solves take too long without this library."""
    if case["family"] == "random" and case["n"] <= 400:
        rp, col, w = (t.cpu().numpy() for t in _graph(case, seed)[:3])
        return _stoer_wagner(case["n"], rp, col, w), None
    if case["family"] == "proposer":
        rp, col, _, second = _graph(case, seed)
        label = np.zeros(rp.numel() - 1)
        label[second.cpu().numpy()] = 1
        loss, grad = _proposer_grad64(rp, col, _proposer_params(seed), label)
        return {"loss": loss, "grad": grad}
    return None
