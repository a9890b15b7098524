// mc_pr.cu -- Padberg-Rinaldi local contraction tests.
//
// The paper cites the tests (Sec. 2.2 related work; used by VieCut,
// Sec. 2.3) without stating them.  With d() the weighted degree of the
// current graph and lam the current bound lambda-hat (always <= delta),
// edge {u, v} of weight c is united when
//   PR1: c >= lam
//   PR2: 2c > min(d(u), d(v))
//   PR3: a common neighbour w has 2(c + c(u,w)) > d(u) and 2(c + c(v,w)) > d(v)
//   PR4: c + sum over common neighbours w of min(c(u,w), c(v,w)) >= lam
// PR1 and PR4 bound lambda(G, u, v) from below by lam (an edge and
// edge-disjoint two-edge paths).  PR2 and PR3 show that any cut below
// delta that separates u and v could be made strictly lighter by moving u
// or v across, so no minimum cut below lambda-hat crosses the edge; the
// strict inequality is what lets all passing edges be contracted at once.
// With level >= 2 a vertex with exactly two neighbours joined by equal
// weights also joins the smaller neighbour: a cut below delta crosses a path
// of such vertices at most once and slides along it at equal weight, and a
// path's k inner vertices close at most k of its k+1 edges.
//
// PR1/PR2: one thread per arc (u < v).  PR3/PR4: one warp per vertex (see
// k_pr34), only on edges whose shorter row has at most `budget` arcs (all
// edges when budget < 0).
#include "mc_internal.cuh"

namespace mc {

__device__ __forceinline__ int row_weight(const int *rp, const int2 *adj, int v, int u) {
    int lo = rp[v], hi = rp[v + 1] - 1;
    while (lo <= hi) {
        int mid = (lo + hi) >> 1;
        int x = adj[mid].x;
        if (x == u) return adj[mid].y;
        if (x < u) lo = mid + 1; else hi = mid - 1;
    }
    return 0;
}

// PR1/PR2 (lo <= 2) on every arc u < v, and the degree-2 tie rule
__global__ void k_pr(const DevGraph g, int *par, long long lam, int lo, int level,
                     unsigned long long *unions) {
    long long local = 0;
    for (i64 j = (i64)blockIdx.x * blockDim.x + threadIdx.x; j < g.arcs; j += (i64)gridDim.x * blockDim.x) {
        const int u = g.src[j];
        const int2 e = g.adj[j];
        const int v = e.x;
        if (u >= v) continue;
        const long long c = e.y;
        const long long du = g.deg[u], dv = g.deg[v];
        bool ok = (lo <= 1 && level >= 1 && c >= lam) ||
                  (lo <= 2 && level >= 2 && 2 * c > (du < dv ? du : dv));
        if (ok && uf_meet<true>(par, u, v, INT_MAX) > 0) ++local;
    }
    // degree-2 tie rule: a vertex with exactly two neighbours of equal weight
    // joins the smaller one (a cut below delta slides along such a path)
    if (lo <= 2 && level >= 2) {
        for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < g.n; u += gridDim.x * blockDim.x) {
            const int a = g.rp[u];
            if (g.rp[u + 1] - a != 2) continue;
            const int2 e0 = g.adj[a], e1 = g.adj[a + 1];
            if (e0.y == e1.y && uf_meet<true>(par, u, e0.x < e1.x ? e0.x : e1.x, INT_MAX) > 0) ++local;
        }
    }
    if (local) atomicAdd(unions, (unsigned long long)local);
}

// PR3/PR4, one warp per vertex u.  Edge {u, v} belongs to the endpoint with
// the shorter row (ties: the smaller id), and only when that row has at most
// `budget` arcs (any length when budget < 0): the warp's lanes take u's
// neighbours w, binary-search c(v, w) in v's sorted row, and the warp sums
// PR4's minima and ORs PR3's condition.  Work per vertex grows with the
// square of its own (short) row, so hubs cost little.  Edges that pass
// PR1/PR2 in the same call (lo <= 2) are left to k_pr.
constexpr int kPrWarps = 8;

__device__ __forceinline__ int find_in_global(const int2 *row, int len, int x) {
    int lo = 0, hi = len - 1;
    while (lo <= hi) {
        const int mid = (lo + hi) >> 1;
        const int2 e = row[mid];
        if (e.x == x) return e.y;
        if (e.x < x) lo = mid + 1; else hi = mid - 1;
    }
    return 0;
}

__global__ void __launch_bounds__(kPrWarps * 32)
k_pr34(const DevGraph g, int *par, long long lam, int lo, int level, int budget, int min_len,
       unsigned long long *unions) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    long long local = 0;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < g.n; u += nw) {
        const int u0 = g.rp[u], u1 = g.rp[u + 1], lu = u1 - u0;
        if (lu <= min_len || (budget >= 0 && lu > budget)) continue;
        const long long du = g.deg[u];
        for (int i0 = u0; i0 < u1; i0 += 32) {
            const int i = i0 + lane;
            bool cand = false;
            int v = 0, c = 0;
            if (i < u1) {
                const int2 e = g.adj[i];
                v = e.x;
                c = e.y;
                const int lv = g.rp[v + 1] - g.rp[v];
                cand = lv > lu || (lv == lu && v > u);
                if (cand && lo <= 2) {
                    const long long dv = g.deg[v];
                    const bool pr12 = (lo <= 1 && level >= 1 && (long long)c >= lam) ||
                                      (level >= 2 && 2LL * c > (du < dv ? du : dv));
                    cand = !pr12;
                }
            }
            unsigned todo = __ballot_sync(0xffffffffu, cand);
            while (todo) {
                const int l = __ffs(todo) - 1;
                todo &= todo - 1;
                const int vv = __shfl_sync(0xffffffffu, v, l);
                const long long cc = __shfl_sync(0xffffffffu, c, l);
                const int v0 = g.rp[vv], lv = g.rp[vv + 1] - v0;
                const long long dv = g.deg[vv];
                long long pr4 = 0;
                bool pr3 = false;
                for (int k = u0 + lane; k < u1; k += 32) {
                    const int2 x = g.adj[k];  // w = x.x, c(u, w) = x.y
                    if (x.x == vv) continue;
                    const int cvw = find_in_global(g.adj + v0, lv, x.x);
                    if (cvw == 0) continue;
                    const long long cuw = x.y;
                    if (2 * (cc + cuw) > du && 2 * (cc + cvw) > dv) pr3 = true;
                    pr4 += cuw < cvw ? cuw : cvw;
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) pr4 += __shfl_xor_sync(0xffffffffu, pr4, o);
                const bool ok = __any_sync(0xffffffffu, pr3) || (level >= 4 && cc + pr4 >= lam);
                if (ok && lane == 0 && uf_meet<true>(par, u, vv, INT_MAX) > 0) ++local;
            }
        }
    }
    if (local) atomicAdd(unions, (unsigned long long)local);
}

// PR3/PR4 for rows of at most kPairRow arcs, one warp per vertex u with
// every (owned edge (u, v), neighbour w of u) pair on its own lane: u's row
// and its owned edges go to shared memory, each lane binary-searches w in
// v's row, and PR4's sums and PR3's flags gather per edge in shared memory.
// The same edges and conditions as k_pr34; a short row fills the warp
// instead of one lane per neighbour.
constexpr int kPairRow = 64;

struct Pr34Smem {
    int w[kPairRow];
    int cw[kPairRow];
    int v[kPairRow];
    int cv[kPairRow];
    int v0[kPairRow];
    int lv[kPairRow];
    long long dv[kPairRow];
    unsigned long long pr4[kPairRow];
    int pr3[kPairRow];
};

__global__ void __launch_bounds__(kPrWarps * 32)
k_pr34_pairs(const DevGraph g, int *par, long long lam, int lo, int level, int max_len,
             unsigned long long *unions) {
    __shared__ Pr34Smem smem[kPrWarps];
    Pr34Smem &sm = smem[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    long long local = 0;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < g.n; u += nw) {
        const int u0 = g.rp[u], lu = g.rp[u + 1] - u0;
        if (lu == 0 || lu > max_len) continue;
        const long long du = g.deg[u];
        // u's row, and the edges u owns (the longer row on the other side,
        // ties to the larger id) that PR1/PR2 do not already take
        int ne = 0;
        for (int i0 = 0; i0 < lu; i0 += 32) {
            const int i = i0 + lane;
            bool own = false;
            int v = 0, c = 0, v0 = 0, lv = 0;
            long long dv = 0;
            if (i < lu) {
                const int2 e = g.adj[u0 + i];
                v = e.x;
                c = e.y;
                sm.w[i] = v;
                sm.cw[i] = c;
                v0 = g.rp[v];
                lv = g.rp[v + 1] - v0;
                dv = g.deg[v];
                own = lv > lu || (lv == lu && v > u);
                if (own && lo <= 2)
                    own = !((lo <= 1 && level >= 1 && (long long)c >= lam) ||
                            (level >= 2 && 2LL * c > (du < dv ? du : dv)));
            }
            const unsigned m = __ballot_sync(0xffffffffu, own);
            if (own) {
                const int j = ne + __popc(m & ((1u << lane) - 1u));
                sm.v[j] = v;
                sm.cv[j] = c;
                sm.v0[j] = v0;
                sm.lv[j] = lv;
                sm.dv[j] = dv;
                sm.pr4[j] = 0;
                sm.pr3[j] = 0;
            }
            ne += __popc(m);
        }
        __syncwarp();
        if (ne == 0) continue;
        const int np = ne * lu;
        for (int p = lane; p < np; p += 32) {
            const int j = p / lu, k = p - j * lu;
            const int x = sm.w[k], vv = sm.v[j];
            if (x == vv) continue;
            const int cvw = find_in_global(g.adj + sm.v0[j], sm.lv[j], x);
            if (cvw == 0) continue;
            const long long cuw = sm.cw[k], cc = sm.cv[j];
            if (2 * (cc + cuw) > du && 2 * (cc + cvw) > sm.dv[j]) sm.pr3[j] = 1;
            atomicAdd(&sm.pr4[j], (unsigned long long)(cuw < cvw ? cuw : cvw));
        }
        __syncwarp();
        for (int j = lane; j < ne; j += 32) {
            const bool ok = sm.pr3[j] != 0 || (level >= 4 && (long long)sm.cv[j] + (long long)sm.pr4[j] >= lam);
            if (ok && uf_meet<true>(par, u, sm.v[j], INT_MAX) > 0) ++local;
        }
        __syncwarp();
    }
    if (local) atomicAdd(unions, (unsigned long long)local);
}

// PR4 (and PR1) on a few arcs of every row.  In a clustered graph almost any
// edge has the common neighbours to pass, and two united edges a vertex leave
// hardly a block of its own, so a few tests a vertex do what otherwise takes a
// scan of every arc: every vertex tests its first arc, then its second if that
// runs between two blocks by then, then one of its first eight that does.
//
// Eight lanes a test: they hold eight arcs of either row, compare them all by
// shuffles, and go on with the next eight of the row whose ids end first, until
// the common weight reaches the bound (or for a number of steps: what is
// counted then is a lower bound, so the test only gets weaker).  Bound by
// latency (offsets, arcs, parents, one after another; issue slots 44 % used)
// and by the neighbours' sectors.  The round against one of concurrent scans,
// hyperbolic graphs: n = 2^20, 34 M arcs, bound 6: 0.88 -> 0.32 ms; n = 2^22,
// 268 M arcs, bound 20: 5.5 -> 2.0 ms.  What was slower: a thread a test (it
// walks the rows one arc at a time, and the lines of a thousand walks a SM push
// each other out of L1: 1.2 ms at n = 2^20); sixteen arcs a step (twice the
// sectors for a bound of 6: the first pass 132 -> 152 us); parents read past L1
// (the common root's word comes from one L2 slice: the last pass 0.63 ms of
// 0.04); tests in place of the job lists (warps with several tests at the end:
// 0.12 ms of 0.02); one atomic a warp on the union counter over a full grid
// (0.28 ms of 0.11).
//
// UNIT: every weight is 1, so a common neighbour counts 1.
struct TriJob {
    int u, v, c;
};

// one test a group of eight lanes (u < 0: none); the common weight, `need` at most
template <bool UNIT>
__device__ __forceinline__ int tri_test(const DevGraph &g, TriJob t, int need, int max_steps) {
    constexpr unsigned kAll = 0xffffffffu;
    const int gl = threadIdx.x & 7;
    const int2 none = make_int2(INT_MAX, 0);
    int i = 0, i1 = 0, j = 0, j1 = 0;
    if (t.u >= 0) {
        i = g.rp[t.u];
        i1 = g.rp[t.u + 1];
        j = g.rp[t.v];
        j1 = g.rp[t.v + 1];
    }
    int2 x = i + gl < i1 ? g.adj[i + gl] : none, y = j + gl < j1 ? g.adj[j + gl] : none;
    int sum = t.c < need ? t.c : need;
    bool act = t.u >= 0 && sum < need;
    for (int st = 0; st < max_steps && __any_sync(kAll, act); ++st) {
        int m;
        if (UNIT) {
            bool h = false;
#pragma unroll
            for (int s = 0; s < 8; ++s) h |= __shfl_sync(kAll, y.x, s, 8) == x.x;
            m = __popc(__ballot_sync(kAll, h && x.x != INT_MAX) & (0xffu << (threadIdx.x & 24)));
        } else {
            int hit = -1;
#pragma unroll
            for (int s = 0; s < 8; ++s)
                if (__shfl_sync(kAll, y.x, s, 8) == x.x) hit = s;
            const int wy = __shfl_sync(kAll, y.y, hit & 7, 8);
            m = hit >= 0 && x.x != INT_MAX ? (x.y < wy ? x.y : wy) : 0;
            m = m < need ? m : need;
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) m += __shfl_xor_sync(kAll, m, o, 8);
        }
        // the row whose ids end first goes on; when it has no more, no common
        // neighbour is left
        const int ex = __shfl_sync(kAll, x.x, i1 - i < 8 ? (i1 - i - 1) & 7 : 7, 8);
        const int ey = __shfl_sync(kAll, y.x, j1 - j < 8 ? (j1 - j - 1) & 7 : 7, 8);
        if (act) {
            sum = m < need - sum ? sum + m : need;
            if (ex <= ey) {
                i += 8;
                act = sum < need && i < i1;
                if (act) x = i + gl < i1 ? g.adj[i + gl] : none;
            } else {
                j += 8;
                act = sum < need && j < j1;
                if (act) y = j + gl < j1 ? g.adj[j + gl] : none;
            }
        }
    }
    return sum;
}

__device__ __forceinline__ void tri_count(int local, unsigned long long *unions) {
    local = (int)__reduce_add_sync(0xffffffffu, (unsigned)local);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(unions, (unsigned long long)local);
}

// every vertex's first arc.  Its end is mostly smaller, and then the vertex
// hangs from it without a find (parents stay smaller than their children).
template <bool UNIT>
__global__ void __launch_bounds__(256, 8)
k_tri_first(const DevGraph g, int *par, int need, int max_steps, unsigned long long *unions) {
    int local = 0;
    for (i64 k = ((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 3; (k & ~3) < g.n; k += (i64)gridDim.x * blockDim.x / 8) {
        const int u = (int)k;
        TriJob t{-1, 0, 0};
        if (u < g.n) {
            const int a = g.rp[u];
            if (a < g.rp[u + 1]) {
                const int2 e = g.adj[a];
                t = TriJob{u, e.x, e.y};
            }
        }
        const int sum = tri_test<UNIT>(g, t, need, max_steps);
        if (t.u >= 0 && sum >= need && (threadIdx.x & 7) == 0) {
            if (t.v < u && atomicCAS(&par[u], u, t.v) == u) ++local;
            else local += uf_meet<true>(par, u, t.v) > 0;
        }
        __syncwarp();
    }
    tri_count(local, unions);
}

// the jobs of the next pass: of each vertex the first of its first eight arcs
// whose end is in another block (parents are roots here); (vertex << 32 | arc)
__global__ void __launch_bounds__(256)
k_tri_collect(const DevGraph g, const int *__restrict__ par, int q1, u64 *jobs, u64 *count) {
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int kV = 4;  // vertices a group of eight lanes looks over at once
    const int lane = threadIdx.x & 31, gl = lane & 7, grp = lane >> 3;
    const int u0 = (int)(((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4 * kV;
    int a0[kV], a1[kV], v[kV], pu[kV];
#pragma unroll
    for (int k = 0; k < kV; ++k) {
        const int u = u0 + 4 * k + grp;
        a0[k] = u < g.n ? g.rp[u] : 0;
        a1[k] = u < g.n ? g.rp[u + 1] : 0;
        pu[k] = u < g.n ? par[u] : -1;
    }
#pragma unroll
    for (int k = 0; k < kV; ++k) v[k] = gl < q1 && a0[k] + gl < a1[k] ? g.adj[a0[k] + gl].x : -1;
    int pos[kV], total = 0;
#pragma unroll
    for (int k = 0; k < kV; ++k) {
        const bool open = v[k] >= 0 && par[v[k]] != pu[k];
        const unsigned mine = (__ballot_sync(kAll, open) >> (lane & 24)) & 0xffu;
        pos[k] = mine ? a0[k] + __ffs(mine) - 1 : -1;
        total += mine != 0u && gl == 0;
    }
    int inc = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kAll, inc, o);
        if (lane >= o) inc += t;
    }
    // one global atomic a block
    __shared__ int wsum[8];
    __shared__ u64 s_base;
    if (lane == 31) wsum[threadIdx.x >> 5] = inc;
    __syncthreads();
    int before = 0;
    for (int w = 0; w < (int)(threadIdx.x >> 5); ++w) before += wsum[w];
    if (threadIdx.x == 255) s_base = before + inc > 0 ? atomicAdd(count, (u64)(before + inc)) : 0;
    __syncthreads();
    u64 base = s_base + (u64)(before + inc - total);
    if (gl == 0) {
#pragma unroll
        for (int k = 0; k < kV; ++k)
            if (pos[k] >= 0) jobs[base++] = ((u64)(u32)(u0 + 4 * k + grp) << 32) | (u32)pos[k];
    }
}

template <bool UNIT>
__global__ void __launch_bounds__(256, 8)
k_tri_jobs(const DevGraph g, int *par, const u64 *__restrict__ jobs, const u64 *count, int need, int max_steps,
           unsigned long long *unions, i64 *tests) {
    const i64 nj = (i64)*count;
    if (blockIdx.x == 0 && threadIdx.x == 0) *tests += nj;
    const i64 step = (i64)gridDim.x * blockDim.x / 8;
    int local = 0;
    for (i64 k0 = ((i64)blockIdx.x * blockDim.x + (threadIdx.x & ~31)) / 8; k0 < nj; k0 += step) {
        const i64 k = k0 + ((threadIdx.x & 31) >> 3);
        TriJob t{-1, 0, 0};
        if (k < nj) {
            const u64 job = jobs[k];
            const int2 e = g.adj[(u32)job];
            t = TriJob{(int)(job >> 32), e.x, e.y};
        }
        const int sum = tri_test<UNIT>(g, t, need, max_steps);
        if (t.u >= 0 && sum >= need && (threadIdx.x & 7) == 0) local += uf_meet<true>(par, t.u, t.v) > 0;
        __syncwarp();
    }
    tri_count(local, unions);
}

template <bool UNIT>
static int launch_triangles(const DevGraph &g, Work &w, int need, cudaStream_t s) {
    const int max_steps = 16 + (need < 4096 ? need : 4096);
    auto *un = reinterpret_cast<unsigned long long *>(&w.st->unions);
    u64 *count = reinterpret_cast<u64 *>(&w.st->count), *jobs = w.keysA;
    int jb = (int)(((i64)g.n * 8 + 255) / 256);
    if (jb > num_sms() * 8) jb = num_sms() * 8;
    ++::mc::g_launches; k_tri_first<UNIT><<<jb, 256, 0, s>>>(g, w.par, need, max_steps, un);
    for (int pass = 0; pass < 2; ++pass) {
        MC_TRY(flatten_parents(w, g.n, s));
        MC_CUDA(cudaMemsetAsync(count, 0, sizeof(u64), s));
        ++::mc::g_launches; k_tri_collect<<<(int)(((i64)g.n * 2 + 255) / 256), 256, 0, s>>>(g, w.par, pass ? 8 : 2, jobs, count);
        ++::mc::g_launches; k_tri_jobs<UNIT><<<jb, 256, 0, s>>>(g, w.par, jobs, count, need, max_steps, un, &w.st->tests);
    }
    return MC_OK;
}

int pr_triangles(const DevGraph &g, Work &w, i64 lam, bool unit, cudaStream_t s) {
    if (lam >= kTriMaxBound || g.arcs == 0) return MC_OK;
    if (unit) MC_TRY(launch_triangles<true>(g, w, (int)lam, s));
    else MC_TRY(launch_triangles<false>(g, w, (int)lam, s));
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

int pr_tests_budget(const DevGraph &g, Work &w, i64 lam, int lo, int level, int budget,
                    cudaStream_t s) {
    if (level <= 0 || lo > level || g.arcs == 0) return MC_OK;
    int blocks = (int)(((g.arcs > g.n ? g.arcs : g.n) + 255) / 256);
    int cap = num_sms() * 16;
    if (blocks > cap) blocks = cap;
    unsigned long long *un = reinterpret_cast<unsigned long long *>(&w.st->unions);
    if (lo <= 2) { ++::mc::g_launches; k_pr<<<blocks, 256, 0, s>>>(g, w.par, lam, lo, level, un); }
    if (level >= 3) {
        long long wb = ((long long)g.n + kPrWarps - 1) / kPrWarps;
        const long long cap = (long long)num_sms() * 8;
        if (wb > cap) wb = cap;
        const int short_len = budget >= 0 && budget < kPairRow ? budget : kPairRow;
        ++::mc::g_launches; k_pr34_pairs<<<(int)wb, kPrWarps * 32, 0, s>>>(g, w.par, lam, lo, level, short_len, un);
        if (budget < 0 || budget > kPairRow) {
            ++::mc::g_launches; k_pr34<<<(int)wb, kPrWarps * 32, 0, s>>>(g, w.par, lam, lo, level, budget, kPairRow, un);
        }
    }
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

}  // namespace mc
