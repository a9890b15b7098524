// mc_dense.cuh -- the last rounds of Alg. 2 on a dense matrix in shared memory.
//
// A contracted graph of at most 224 vertices fits one block's shared memory as
// a matrix of 32-bit weights (clamped at the bound as everywhere).  One warp
// then scans it (Alg. 3): a lane owns every 32nd column -- its r-value and join
// in registers -- so that a pop is a load of the popped row, an update a column
// and one warp maximum over (key, vertex) words, with no queue and no list of
// arcs.  The whole block does what surrounds the scan: PR1/PR2 and the degree-2
// rule, the unions, the contraction (rows added up in place, a thread a column,
// then columns, a warp a row) and the degrees.
//
// The rounds, their start vertices, the order of pops (the smallest vertex of
// the largest key) and so every result are those of the single-warp solver
// over lists (mc_batch.cu, k_tail), which larger graphs and bounds keep.
// Bound by the scan's chain of dependent instructions: about 370 cycles a pop
// at 200 vertices, against 1170 to 2000.  200 vertices, 1154 edges, weights to
// 100: 193 -> 58 us with the read of the result (46 us the kernel); the 76
// vertices left of RHG 2^20: 100 -> 40 us.  Eight neighbouring 16-bit columns a
// lane, one load a pop, took 490 cycles: what it saves in loads it spends on
// taking the columns apart and the popped vertex out.
#pragma once

#include "mc_internal.cuh"

namespace mc {

namespace dense {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr unsigned kAll = 0xffffffffu;
constexpr int kSelf = -(1 << 30);  // on the diagonal: takes a vertex out as it is popped

// N = the most vertices: a lane owns N / 32 columns at most, a thread one
template <int N>
struct DenseSmem {
    static constexpr int kN = N;
    static_assert(N % 32 == 0 && N <= kDenseN && N <= kThreads, "");
    int M[kN * kN];  // rows of kN
    unsigned acc[kWarps][kN];
    int par[kThreads], deg[kN], lab[kThreads], joinx[kN], first[kThreads + 1], cursor[kThreads], r[kN];
    unsigned short perm[kN], orig[kThreads], order[kN];
    u32 best[kWarps];
    int wsum[kWarps];
    i64 lam;
    int un, len, arg;
};

// the block's first 256 threads (a kernel with more runs the rest by)
__device__ __forceinline__ void sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

__device__ __forceinline__ int sm_find(int *par, int x) {
    volatile int *p = par;
    while (true) {
        const int q = p[x];
        if (q == x) return x;
        x = q;
    }
}

__device__ __forceinline__ bool sm_union(int *par, int a, int b) {
    while (true) {
        a = sm_find(par, a);
        b = sm_find(par, b);
        if (a == b) return false;
        if (a > b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(&par[b], b, a) == b) return true;
    }
}

// exclusive scan of one flag a thread; *total = the sum (all threads call)
__device__ __forceinline__ int block_rank(bool flag, int *wsum, int *total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const unsigned m = __ballot_sync(kAll, flag);
    if (lane == 0) wsum[wid] = __popc(m);
    sync();
    int before = 0, sum = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
        before += w < wid ? wsum[w] : 0;
        sum += wsum[w];
    }
    *total = sum;
    sync();
    return before + __popc(m & ((1u << lane) - 1u));
}

// the minimum degree below s.lam, if there is one, becomes the bound, with the
// smallest such vertex as its side (n0 = vertices of the input)
template <int N>
__device__ inline void take_min_degree(DenseSmem<N> &s, int n, int n0) {
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid < 32) {
        int d = INT_MAX, arg = 0;
        for (int v = lane; v < n; v += 32)
            if (s.deg[v] < d) {
                d = s.deg[v];
                arg = v;
            }
        const int md = (int)__reduce_min_sync(kAll, (unsigned)d);
        arg = (int)__reduce_min_sync(kAll, d == md ? (unsigned)arg : kAll);
        if (lane == 0) {
            s.arg = md < s.lam ? arg : -1;
            if (md < s.lam) s.lam = md;
        }
    }
    sync();
    if (s.arg >= 0) {
        const unsigned m = __ballot_sync(kAll, tid < n0 && s.orig[tid] == s.arg);
        if (lane == 0) s.best[tid >> 5] = m;
    }
    sync();
}

// One capped scan (Alg. 3) by warp 0; a lane owns columns lane, lane + 32, ..,
// KC of them.  A queue entry is min(r, C) << 8 | 255 - v: a vertex not reached
// (r = 0) stays below 256, one popped (r far below 0, its key -1) below 0, and
// no update needs to know which it was.  The next pop depends on the updates
// alone; alpha and the joins follow while the maximum is on its way.
template <int KC, int N>
__device__ inline void dense_scan(DenseSmem<N> &s, int n, int start) {
    constexpr int kN = N;
    const int lane = threadIdx.x;
    const int C = (int)s.lam;
    int r[KC], jx[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) {
        r[k] = 0;
        jx[k] = -1;
        s.r[32 * k + lane] = 0;
        s.order[32 * k + lane] = 0xffff;
    }
    __syncwarp();
    i64 L = C, alpha = 0;
    int Lj = C, nS = 0, len = 0, p = start;
    while (true) {
        int c[KC], e[KC];
#pragma unroll
        for (int k = 0; k < KC; ++k) c[k] = s.M[p * kN + 32 * k + lane];
        const int dp = s.deg[p], rx = s.r[p];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < KC; ++k) {
            r[k] += c[k];
            s.r[32 * k + lane] = r[k];
            const int key = r[k] < C ? (r[k] > -1 ? r[k] : -1) : C;
            e[k] = key * 256 + (255 - 32 * k - lane);
        }
        __syncwarp();  // the next pop's r comes from another lane's store
#pragma unroll
        for (int o = 1; o < KC; o *= 2)
#pragma unroll
            for (int k = 0; k + o < KC; k += 2 * o) e[k] = e[k] > e[k + o] ? e[k] : e[k + o];
        const int top = __reduce_max_sync(kAll, e[0]);
        if (lane == 0) s.order[p] = (unsigned short)nS;
        ++nS;
        alpha += dp - 2LL * rx;
        if (alpha < L && nS < n) {
            L = alpha;
            Lj = (int)alpha;
            len = nS;
        }
#pragma unroll
        for (int k = 0; k < KC; ++k)
            if (r[k] >= Lj && r[k] - c[k] < Lj) jx[k] = p;
        if (top < 256) break;
        p = 255 - (top & 255);
    }
#pragma unroll
    for (int k = 0; k < KC; ++k) s.joinx[32 * k + lane] = jx[k];
    if (lane == 0) {
        s.len = L < C ? len : 0;
        s.lam = L;
    }
}

template <int N>
__device__ __forceinline__ void scan(DenseSmem<N> &s, int n, int start) {
    const int kc = (n + 31) / 32;
    if (kc == 1) return dense_scan<1>(s, n, start);
    if constexpr (N >= 64)
        if (kc == 2) return dense_scan<2>(s, n, start);
    if constexpr (N >= 96)
        if (kc == 3) return dense_scan<3>(s, n, start);
    if constexpr (N >= 128)
        if (kc == 4) return dense_scan<4>(s, n, start);
    if constexpr (N >= 160)
        if (kc == 5) return dense_scan<5>(s, n, start);
    if constexpr (N >= 192)
        if (kc == 6) return dense_scan<6>(s, n, start);
    if constexpr (N >= 224) return dense_scan<7>(s, n, start);
}

// the rounds on the graph in s.M, s.deg, s.orig (n0 vertices, orig the
// identity) under the bound s.lam, which they lower, with the side in s.best;
// an error code.  Threads 0 .. 255 of the block call.
template <int N>
__device__ inline int rounds(DenseSmem<N> &s, int n0, u64 seed, int pr_level) {
    constexpr int kN = N;
    int *M = s.M;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    int n = n0, err = 0;
    int round = 0, guard = 0;
    while (n >= 2 && s.lam > 0) {
        if (++guard > 4 * n0 + 16) { err = MC_EINTERNAL; break; }
        const i64 lam = s.lam;
        s.par[tid] = tid;
        if (tid == 0) s.un = 0;
        sync();
        // PR1/PR2 and the degree-2 rule, a warp a row (warp 0 scans meanwhile)
        int un = 0;
        if (pr_level >= 1 && wid > 0) {
            for (int u = wid - 1; u < n; u += kWarps - 1) {
                const int du = s.deg[u];
                int cnt = 0, va = 0, vb = 0;  // the first two neighbours
                for (int v0 = 0; v0 < n; v0 += 32) {
                    const int v = v0 + lane;
                    const int c = v < n ? M[u * kN + v] : 0;
                    if (c > 0 && v > u) {
                        const int dv = s.deg[v];
                        if (c >= lam || (pr_level >= 2 && 2 * c > (du < dv ? du : dv))) un += sm_union(s.par, u, v);
                    }
                    unsigned m = __ballot_sync(kAll, c > 0);
                    while (m && cnt < 3) {
                        const int x = v0 + __ffs(m) - 1;
                        m &= m - 1u;
                        if (cnt == 0) va = x;
                        if (cnt == 1) vb = x;
                        ++cnt;
                    }
                }
                if (pr_level >= 2 && cnt == 2 && lane == 0 && M[u * kN + va] == M[u * kN + vb])
                    un += sm_union(s.par, u, va);
            }
        }
        // one scan; its joins
        if (wid == 0) {
            const u64 h = splitmix64(seed ^ splitmix64((0x7A11ULL << 20) ^ (u64)round));
            scan(s, n, (int)(h % (u64)n));
        }
        sync();
        if (tid < n && s.joinx[tid] >= 0) un += sm_union(s.par, s.joinx[tid], tid);
        if (un) atomicAdd(&s.un, un);
        sync();
        ++round;
        if (s.lam < lam) {
            const int len = s.len;
            const unsigned m = __ballot_sync(kAll, tid < n0 && s.order[s.orig[tid < n0 ? tid : 0]] < len);
            if (lane == 0) s.best[wid] = m;
            if (s.un == 0) {
                sync();
                continue;
            }
        }
        if (s.un == 0) { err = MC_EINTERNAL; break; }
        // number the blocks by their smallest members; the members in block order
        const int root = tid < n ? sm_find(s.par, tid) : -1;
        int nc = 0;
        const int rank = block_rank(root == tid, s.wsum, &nc);
        if (root == tid) s.lab[tid] = rank;
        s.cursor[tid] = 0;
        sync();
        const int mine = tid < n ? s.lab[root] : 0;
        sync();
        if (tid < n) {
            s.lab[tid] = mine;
            atomicAdd(&s.cursor[mine], 1);
        }
        sync();
        if (wid == 0) {
            int carry = 0;
            for (int b0 = 0; b0 < kThreads; b0 += 32) {
                const int v = s.cursor[b0 + lane];
                int inc = v;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(kAll, inc, o);
                    if (lane >= o) inc += t;
                }
                s.first[b0 + lane] = carry + inc - v;
                s.cursor[b0 + lane] = carry + inc - v;
                carry += __shfl_sync(kAll, inc, 31);
            }
            if (lane == 0) s.first[kThreads] = carry;
        }
        sync();
        if (tid < n) s.perm[atomicAdd(&s.cursor[mine], 1)] = (unsigned short)tid;
        sync();
        // rows: block a's members lie at a or later, so its sum may take row a
        const int cap = (int)s.lam;
        if (tid < n) {
            for (int a = 0; a < nc; ++a) {
                int sum = 0;
                for (int i = s.first[a]; i < s.first[a + 1]; ++i) sum += M[s.perm[i] * kN + tid];
                M[a * kN + tid] = sum < cap ? sum : cap;
            }
        }
        sync();
        // columns, and the degrees
        unsigned *acc = s.acc[wid];
        for (int a = wid; a < nc; a += kWarps) {
            for (int v = lane; v < n; v += 32) {
                const int c = M[a * kN + v], b = s.lab[v];
                if (c > 0 && b != a) atomicAdd(&acc[b], (unsigned)c);
            }
            __syncwarp();
            int d = 0;
            for (int b = lane; b < n; b += 32) {
                const unsigned x = acc[b];
                const int c = x < (unsigned)cap ? (int)x : cap;
                acc[b] = 0;
                M[a * kN + b] = b == a ? kSelf : c;
                d += c;
            }
            d = (int)__reduce_add_sync(kAll, (unsigned)d);
            if (lane == 0) s.deg[a] = d;
            __syncwarp();
        }
        if (tid < n0) s.orig[tid] = (unsigned short)s.lab[s.orig[tid]];
        n = nc;
        sync();
        if (n >= 2) take_min_degree(s, n, n0);
    }
    sync();
    return err;
}

}  // namespace dense

}  // namespace mc
