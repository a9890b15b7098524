// mc_batch_cta.cu -- many independent graphs at once, one block per graph.
//
// The warp-per-graph solver (mc_batch.cu) spends its time in one chain: a scan
// of a thousand pops or more, each waiting for the one before it, while the
// largest graphs of a batch keep the launch waiting for theirs.  Here a block
// takes a graph through rounds of forest packing (the certificate of
// mc_forest.cu) in shared memory instead:
//   * the arcs are read from the input in place, checked (canonical rows, every
//     arc with its mirror) and the edges staged as 16-bit ends and weights;
//   * a round packs T <= kMaxT forests over the current blocks, 16-bit parents
//     each.  With a bound above T the edges count in units of s = ceil(bound /
//     T), floor(c / s) of them, which certifies no less than s * T >= bound.  An
//     edge goes into the first forest that has its ends apart (the forests
//     nest, so a binary search finds it) and the next as long as it has units;
//     one with a unit to spare after all of them unites its ends;
//   * a contraction only relabels: parallel edges and edges inside a block do
//     no harm to the packing, so the staged edges stay as they are;
//   * the last kDN blocks' weights are added up in a matrix and the dense
//     rounds (mc_dense.cuh) finish.
// A graph this does not suit (too large, rows not canonical, a round that
// unites little, any error) goes to a list that the warp-per-graph solver
// works off afterwards, so results and errors are that solver's.
//
// Bound by the latency of shared memory and of the three reads of the arcs; to
// hide it a SM holds 1024 threads whatever the graphs: four blocks of 256, two
// of 512 or one of 1024, the smallest share of shared memory that holds the
// graph.  What is left is the packing's walks, 11 of 32 lanes busy on average.
// 4096 graphs of 50 to 2000 vertices, mean degree 4 to 16, weights to 100: 4.1 ms
// with a warp a graph, 1.8 so (2.8 with 16 forests always and a search of the
// offsets for every arc's row); 96 graphs of 50 to 400: 0.6 and 0.16; 1216
// graphs of 2000, weights of 1: 4.5 and 0.81.
#include <algorithm>

#include "mc_batch_cta.cuh"
#include "mc_dense.cuh"

namespace mc {

namespace {

// forests: kShare times the bound over the mean degree (random graphs: 32 costs
// no more rounds and leaves about as many blocks as 16 forests always, at a
// third of the work), between 3 and kMaxT; kManyT after a poor round
constexpr int kShare = 32, kMaxT = 16, kManyT = 64;
constexpr int kMinT = 8;       // no room for more: the rounding would lose too much of the weights
constexpr int kMaxW = 0x7fff;  // sums over the edges that fit stay below 2^31
constexpr int kDN = 64;        // blocks the matrix holds
constexpr int kFew = 32;       // blocks it takes over at, however well the rounds do
constexpr unsigned kAll = 0xffffffffu;
using Dense = dense::DenseSmem<kDN>;

struct CtaSmem {
    u32 best[kCtaMaxN / 32];
    int wsum[32];
    int un, md, arg, graph, cross;
    unsigned tot;
};

// a graph's arrays behind CtaSmem, in bytes from its end
struct CtaLayout {
    int rp, up, uoff, bits, cnt, lab, e, more;
};
__host__ __device__ inline CtaLayout cta_layout(int n, int E) {
    CtaLayout L;
    int at = 0;
    L.rp = at;
    at += 4 * (n + 1);
    L.up = at;  // later the degrees
    at += 4 * n;
    L.uoff = at;  // later the last forest
    at += 4 * (n + 1);
    L.bits = at;
    at += 4 * (E / 16 + 1);
    L.cnt = at;
    at += 2 * (E / 16 + 1);
    L.lab = at;
    at += 2 * n;
    L.e = at;
    at += 6 * E;
    L.more = (at + 15) & ~15;
    return L;
}
__host__ __device__ inline int cta_bytes(int n, int E, int T) {
    const int f = 2 * n * (T - 1), d = (int)sizeof(Dense);
    return (int)sizeof(CtaSmem) + 16 + cta_layout(n, E).more + (f > d ? f : d);
}

constexpr int kSmem[kCtaClasses] = {227 * 1024, 113 * 1024, 56 * 1024};
constexpr int kThreadsOf[kCtaClasses] = {1024, 512, 256};

// the row of arc i: rows that start at or before it, a bit an arc and a count a
// word (the lanes of a warp read one word; a search of the offsets took eleven
// dependent loads an arc)
__device__ __forceinline__ int row_of(const u32 *bits, const unsigned short *cnt, int i) {
    return (int)cnt[i >> 5] + __popc(bits[i >> 5] << (31 - (i & 31))) - 1;
}

// exclusive scan over the block of one value a thread; *total = the sum
template <int TH>
__device__ int cta_scan(int v, int *wsum, int *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kAll, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) wsum[wid] = inc;
    __syncthreads();
    int before = 0, sum = 0;
#pragma unroll
    for (int k = 0; k < TH / 32; ++k) {
        before += k < wid ? wsum[k] : 0;
        sum += wsum[k];
    }
    __syncthreads();
    *total = sum;
    return before + inc - v;
}

// Both ends walk up, the one with the larger parent first: parents are smaller
// than their children, so when that one is a root the ends are apart.  UNITE
// links it.  True if the ends are (were) connected.
template <bool UNITE>
__device__ __forceinline__ bool meet16(unsigned short *par, int a, int b) {
    volatile unsigned short *p = par;
    int pa = p[a], pb = p[b];
    while (true) {
        if (pa == pb) return true;
        if (pa < pb) {
            int t = a; a = b; b = t;
            t = pa; pa = pb; pb = t;
        }
        if (pa == a) {
            if (!UNITE) return false;
            const int old = atomicCAS(par + a, (unsigned short)a, (unsigned short)pb);
            if (old == a) return false;
            pa = old;
            continue;
        }
        const int ga = p[pa];
        if (ga != pa) p[a] = (unsigned short)ga;
        a = pa;
        pa = ga;
    }
}

// the side of the vertices f is true for
template <int TH, class F>
__device__ void cta_side(CtaSmem &s, int n, F f) {
    const int lane = threadIdx.x & 31;
    for (int w = threadIdx.x >> 5; w < (n + 31) / 32; w += TH / 32) {
        const int v = 32 * w + lane;
        const unsigned m = __ballot_sync(kAll, v < n && f(v));
        if (lane == 0) s.best[w] = m;
    }
}

// The rule for degree 2 (mc_pr.cu) on the blocks: one with exactly two edges
// out, of equal weight, goes with the end of one of them.  A packing unites two
// vertices of a cycle a round, and a cycle given up went through the warps after
// all: 300 cycles of 200 to 1100 vertices 3.2 ms a call, 0.21 so (2.8 by the warps
// alone).  Returns the unions; x: 3 nb ints.
template <int TH>
__device__ int cta_paths(CtaSmem &s, const unsigned short *lab, const unsigned short *ua, const unsigned short *va,
                         const unsigned short *wa, int E, int nb, unsigned short *par, int *x) {
    int *cnt = x, *diff = x + nb, *pick = x + 2 * nb;
    __syncthreads();  // s.un has been read
    for (int b = threadIdx.x; b < nb; b += TH) {
        cnt[b] = 0;
        diff[b] = 0;
        pick[b] = INT_MAX;
    }
    if (threadIdx.x == 0) s.un = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < E; e += TH) {
        const int a = lab[ua[e]], b = lab[va[e]], w = wa[e];
        if (a == b) continue;
        atomicAdd(&cnt[a], 1);
        atomicAdd(&cnt[b], 1);
        atomicXor(&diff[a], w);
        atomicXor(&diff[b], w);
        atomicMin(&pick[a], e);
        atomicMin(&pick[b], e);
    }
    __syncthreads();
    int un = 0;
    for (int e = threadIdx.x; e < E; e += TH) {
        const int a = lab[ua[e]], b = lab[va[e]];
        if (a == b) continue;
        const bool take = (cnt[a] == 2 && diff[a] == 0 && pick[a] == e) || (cnt[b] == 2 && diff[b] == 0 && pick[b] == e);
        if (take && !meet16<true>(par, a, b)) ++un;
    }
    un = (int)__reduce_add_sync(kAll, (unsigned)un);
    if ((threadIdx.x & 31) == 0 && un) atomicAdd(&s.un, un);
    __syncthreads();
    return s.un;
}

// one graph; false = left to the warp-per-graph solver.  All threads call, and
// agree on what they return.
template <int TH>
__device__ bool cta_solve(const CtaBatch &B, int gi, CtaSmem &s, unsigned char *data, int bytes) {
    constexpr int kPer = (kCtaMaxN + TH - 1) / TH;  // vertices a thread numbers
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const long long v0 = B.voff[gi];
    const int n = (int)(B.voff[gi + 1] - v0);
    const int *rp_in = B.rp + v0 + gi;
    const long long arc0 = B.aoff[gi];
    const int m = (int)(B.aoff[gi + 1] - arc0), E = m / 2;
    const int *col = B.col + arc0, *wt = B.w + arc0;
    const CtaLayout L = cta_layout(n, E);
    int *rp = reinterpret_cast<int *>(data + L.rp), *up = reinterpret_cast<int *>(data + L.up),
        *uoff = reinterpret_cast<int *>(data + L.uoff);
    u32 *bits = reinterpret_cast<u32 *>(data + L.bits);
    unsigned short *cnt = reinterpret_cast<unsigned short *>(data + L.cnt);
    unsigned short *lab = reinterpret_cast<unsigned short *>(data + L.lab),
                   *ua = reinterpret_cast<unsigned short *>(data + L.e), *va = ua + E, *wa = va + E;

    // offsets: from 0 to m, rising (a graph with an empty row is not connected,
    // and left to the other solver)
    const int words = E / 16 + 1;
    bool bad = 2 * E != m;
    for (int i = tid; i < words; i += TH) bits[i] = 0;
    for (int v = tid; v <= n; v += TH) {
        const int r = rp_in[v];
        rp[v] = r;
        if (r < 0 || r > m || (v == 0 ? r != 0 : rp_in[v - 1] >= r) || (v == n && r != m)) bad = true;
    }
    if (__syncthreads_or(bad)) return false;
    for (int v = tid; v < n; v += TH) atomicOr(&bits[rp[v] >> 5], 1u << (rp[v] & 31));

    // each row's first arc to a larger vertex (rows increase, or the next pass says not)
    int lo[kPer], hi[kPer], found = 0;
    bool more = false;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int v = tid * kPer + k;
        lo[k] = v < n ? rp[v] : 0;
        hi[k] = v < n ? rp[v + 1] : 0;
        more |= lo[k] < hi[k];
    }
    while (more) {
        more = false;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            if (lo[k] < hi[k]) {
                const int mid = (lo[k] + hi[k]) >> 1;
                if (col[mid] > tid * kPer + k) hi[k] = mid;
                else lo[k] = mid + 1;
                more |= lo[k] < hi[k];
            }
        }
    }
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int v = tid * kPer + k;
        if (v < n) {
            up[v] = lo[k];
            found += rp[v + 1] - lo[k];
        }
    }
    int total = 0, at0 = cta_scan<TH>(found, s.wsum, &total);
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        const int v = tid * kPer + k;
        if (v < n) {
            uoff[v] = at0;
            at0 += rp[v + 1] - lo[k];
        }
    }
    if (tid == 0) uoff[n] = total;
    if (total != E) return false;
    // the counts of the words before
    constexpr int kWordsPer = kCtaMaxM / 32 / TH + 1;
    int mine = 0, all = 0;
    for (int k = 0; k < kWordsPer; ++k) {
        const int i = tid * kWordsPer + k;
        if (i < words) mine += __popc(bits[i]);
    }
    int before = cta_scan<TH>(mine, s.wsum, &all);
    for (int k = 0; k < kWordsPer; ++k) {
        const int i = tid * kWordsPer + k;
        if (i < words) {
            cnt[i] = (unsigned short)before;
            before += __popc(bits[i]);
        }
    }
    __syncthreads();
    // rows: increasing, in range, no loop, weights of 15 bits; the edges staged
#pragma unroll 4
    for (int i = tid; i < m; i += TH) {
        const int c = col[i], w = wt[i], prev = i > 0 ? col[i - 1] : -1;
        const int u = row_of(bits, cnt, i), first = up[u];
        if (c < 0 || c >= n || c == u || w <= 0 || w > kMaxW || (!((bits[i >> 5] >> (i & 31)) & 1u) && prev >= c) || (c > u) != (i >= first)) {
            bad = true;
        } else if (c > u) {
            const int at = uoff[u] + i - first;
            ua[at] = (unsigned short)u;
            va[at] = (unsigned short)c;
            wa[at] = (unsigned short)w;
        }
    }
    if (__syncthreads_or(bad)) return false;
    // symmetry: every arc down finds its edge, and there are as many as edges
#pragma unroll 2
    for (int i = tid; i < m; i += TH) {
        const int c = col[i], w = wt[i], u = row_of(bits, cnt, i);
        if (c < u) {
            int lo = uoff[c], hi = uoff[c + 1] - 1;
            bool found = false;
            while (lo <= hi) {
                const int mid = (lo + hi) >> 1, x = va[mid];
                if (x == u) {
                    found = wa[mid] == w;
                    break;
                }
                if (x < u) lo = mid + 1;
                else hi = mid - 1;
            }
            if (!found) bad = true;
        }
    }
    for (int v = tid; v < n; v += TH) lab[v] = (unsigned short)v;
    if (__syncthreads_or(bad)) return false;

    // rounds
    int *deg = up;
    unsigned short *par = reinterpret_cast<unsigned short *>(uoff), *F = reinterpret_cast<unsigned short *>(data + L.more);
    const int room = (bytes - L.more) / 2;  // 16-bit parents F may hold
    int nb = n;
    bool poor = false;
    i64 lam = LLONG_MAX;
    while (true) {
        for (int b = tid; b < nb; b += TH) deg[b] = 0;
        if (tid == 0) {
            s.md = INT_MAX;
            s.arg = INT_MAX;
            s.un = 0;
            s.tot = 0;
            s.cross = 0;
        }
        __syncthreads();
        int cross = 0;
#pragma unroll 4
        for (int e = tid; e < E; e += TH) {
            const int a = lab[ua[e]], b = lab[va[e]], w = wa[e];
            if (a != b) {
                ++cross;
                atomicAdd(&deg[a], w);
                atomicAdd(&deg[b], w);
            }
        }
        cross = (int)__reduce_add_sync(kAll, (unsigned)cross);
        if (lane == 0 && cross) atomicAdd(&s.cross, cross);
        __syncthreads();
        int d = INT_MAX;
        unsigned tot = 0;
        for (int b = tid; b < nb; b += TH) {
            d = deg[b] < d ? deg[b] : d;
            tot += (unsigned)deg[b];
        }
        d = (int)__reduce_min_sync(kAll, (unsigned)d);
        tot = __reduce_add_sync(kAll, tot);
        if (lane == 0) {
            atomicMin(&s.md, d);
            atomicAdd(&s.tot, tot);
        }
        __syncthreads();
        const int md = s.md;
        if (md < lam) {
            for (int b = tid; b < nb; b += TH)
                if (deg[b] == md) atomicMin(&s.arg, b);
            __syncthreads();
            const int arg = s.arg;
            cta_side<TH>(s, n, [&](int v) { return lab[v] == arg; });
            lam = md;
        }
        if (lam == 0 || nb <= kFew) break;
        // forests: more the closer the bound is to the mean degree, as many as fit
        int T = room / nb + 1;
        if (T < kMinT && T < lam) return false;
        // (and units of at most the mean weight: a weight below one counts nothing)
        const i64 share = kShare * nb > 2 * s.cross ? kShare * nb : 2 * s.cross;
        const i64 want = (share * lam + s.tot - 1) / s.tot;
        const int most = poor ? kManyT : want < 3 ? 3 : want < kMaxT ? (int)want : kMaxT;
        T = T < most ? T : most;
        T = lam < T ? (int)lam : T;
        const int unit = (int)((lam + T - 1) / T);
        T = (int)((lam + unit - 1) / unit);
        const int L = T - 1;  // the last is par
        for (int b = tid; b < nb; b += TH) {
            par[b] = (unsigned short)b;
            for (int j = 0; j < L; ++j) F[j * nb + b] = (unsigned short)b;
        }
        __syncthreads();
        int un = 0;
        for (int e = tid; e < E; e += TH) {
            const int a = lab[ua[e]], b = lab[va[e]];
            int c = wa[e] / unit;
            if (a == b || c == 0 || meet16<false>(par, a, b)) continue;
            int lo = 0, hi = L;  // the first forest that has them apart
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (meet16<false>(F + mid * nb, a, b)) lo = mid + 1;
                else hi = mid;
            }
            for (; lo < L && c > 0; ++lo)
                if (!meet16<true>(F + lo * nb, a, b)) --c;
            if (c > 0 && !meet16<true>(par, a, b)) ++un;
        }
        un = (int)__reduce_add_sync(kAll, (unsigned)un);
        if (lane == 0 && un) atomicAdd(&s.un, un);
        __syncthreads();
        const int united = s.un;
        if (united * 8 < nb) {
            // more forests lose less of the weights
            if (!poor && T < kManyT && lam > T) {
                poor = true;
                if (united == 0) continue;
            } else if (nb <= kDN) {
                break;
            } else if (B.pr_level < 2 || cta_paths<TH>(s, lab, ua, va, wa, E, nb, par, reinterpret_cast<int *>(F)) * 8 < nb) {
                return false;
            }
        }
        // number the blocks (in deg) by their smallest members
        int root[kPer], cnt = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int b = tid * kPer + k;
            root[k] = -1;
            if (b < nb) {
                int x = b;
                while (par[x] != x) x = par[x];
                root[k] = x;
                cnt += x == b;
            }
        }
        int total = 0;
        int at = cta_scan<TH>(cnt, s.wsum, &total);
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int b = tid * kPer + k;
            if (root[k] == b) deg[b] = at++;
        }
        __syncthreads();
        int id[kPer];
#pragma unroll
        for (int k = 0; k < kPer; ++k) id[k] = root[k] >= 0 ? deg[root[k]] : 0;
        __syncthreads();
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            const int b = tid * kPer + k;
            if (b < nb) deg[b] = id[k];
        }
        __syncthreads();
        for (int v = tid; v < n; v += TH) lab[v] = (unsigned short)deg[lab[v]];
        __syncthreads();
        nb = total;
        if (nb < 2) break;
    }
    __syncthreads();
    if (lam > 0 && nb >= 2) {
        if (lam > kDenseMaxLam) return false;
        Dense &D = *reinterpret_cast<Dense *>(F);
        int *M = D.M;
        for (int i = tid; i < nb * kDN / 4; i += TH) reinterpret_cast<int4 *>(M)[i] = make_int4(0, 0, 0, 0);
        for (int i = tid; i < dense::kWarps * kDN; i += TH) (&D.acc[0][0])[i] = 0;
        if (tid < dense::kThreads) D.orig[tid] = (unsigned short)tid;
        if (tid == 0) D.lam = lam;
        __syncthreads();
        for (int e = tid; e < E; e += TH) {
            const int a = lab[ua[e]], b = lab[va[e]], w = wa[e];
            if (a != b) {
                atomicAdd(&M[a * kDN + b], w);
                atomicAdd(&M[b * kDN + a], w);
            }
        }
        __syncthreads();
        for (int a = wid; a < nb; a += (TH / 32)) {
            int d = 0;
            for (int b = lane; b < nb; b += 32) {
                const int c = M[a * kDN + b] < lam ? M[a * kDN + b] : (int)lam;
                M[a * kDN + b] = b == a ? dense::kSelf : c;
                d += c;
            }
            d = (int)__reduce_add_sync(kAll, (unsigned)d);
            if (lane == 0) D.deg[a] = d;
        }
        __syncthreads();
        bad = tid < dense::kThreads && dense::rounds(D, nb, B.seed ^ (u64)gi, B.pr_level) != MC_OK;
        if (__syncthreads_or(bad)) return false;
        if (D.lam < lam) {
            lam = D.lam;
            cta_side<TH>(s, n, [&](int v) { return (D.best[lab[v] >> 5] >> (lab[v] & 31)) & 1u; });
        }
        __syncthreads();
    }
    if (tid == 0) {
        B.lam_out[gi] = lam;
        B.err_out[gi] = 0;
    }
    if (B.bits_out) {
        u32 *dst = B.bits_out + B.bits_off[gi];
        const int nw = (n + 31) / 32;
        const bool flip = s.best[0] & 1u;
        for (int i = tid; i < nw; i += TH) {
            u32 x = flip ? ~s.best[i] : s.best[i];
            if (i == nw - 1 && (n & 31)) x &= (1u << (n & 31)) - 1u;
            dst[i] = x;
        }
    }
    return true;
}

template <int C>
__global__ void __launch_bounds__(kThreadsOf[C], 1024 / kThreadsOf[C]) k_batch_cta(CtaBatch B) {
    extern __shared__ __align__(16) unsigned char raw[];
    CtaSmem &s = *reinterpret_cast<CtaSmem *>(raw);
    constexpr int kThreads = kThreadsOf[C], kBytes = kSmem[C];
    constexpr int kHead = (sizeof(CtaSmem) + 15) & ~15;
    while (true) {
        __syncthreads();
        if (threadIdx.x == 0) s.graph = atomicAdd(B.next + C, 1);
        __syncthreads();
        const int k = s.graph;
        if (k >= B.count[C]) break;
        const int gi = B.order[B.first[C] + k];
        if (!cta_solve<kThreads>(B, gi, s, raw + kHead, kBytes - kHead)) {
            __syncthreads();
            if (threadIdx.x == 0) B.rest[atomicAdd(B.nrest, 1)] = gi;
        }
    }
}

template <int C>
int launch_class(const CtaBatch &B, cudaStream_t s) {
    if (B.count[C] == 0) return MC_OK;
    MC_CUDA(cudaFuncSetAttribute(k_batch_cta<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem[C]));
    const int blocks = std::min(B.count[C], num_sms() * (1024 / kThreadsOf[C]));
    ++::mc::g_launches; k_batch_cta<C><<<blocks, kThreadsOf[C], kSmem[C], s>>>(B);
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

}  // namespace

int batch_cta_class(int n, long long m) {
    if (n < 2 || n > kCtaMaxN || m > kCtaMaxM) return -1;
    for (int c = kCtaClasses - 1; c >= 0; --c)
        if (cta_bytes(n, (int)m / 2, c == 0 ? kMinT : kMaxT) <= kSmem[c]) return c;
    return -1;
}

bool batch_cta_chain(int n) { return n > kFew && n < kCtaChainN; }

int batch_cta_launch(const CtaBatch &B, const cudaStream_t (&s)[kCtaClasses]) {
    static_assert(kCtaClasses == 3, "");
    MC_TRY(launch_class<0>(B, s[0]));
    MC_TRY(launch_class<1>(B, s[1]));
    return launch_class<2>(B, s[2]);
}

}  // namespace mc
