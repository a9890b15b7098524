// mc_forest.cu -- a round of connectivity certificates by forest packing.
//
// A scan of CAPFOREST (Alg. 3) unites two vertices once it has seen lambda-hat
// edge-disjoint ways between them, and it sees them one pop after another.
// Edge-disjoint spanning forests certify the same, in the manner of Nagamochi
// and Ibaraki's sparse certificates, without an order: vertices connected in
// each of t forests that share no edge have t edge-disjoint paths between
// them, one in each, so with t = lambda-hat they are united.  An edge of
// weight c is c parallel unit edges, each of which may lie in a forest of its
// own.
//
// The forests start without a single union: in forest j every vertex hangs
// from the end of its j-th unit of weight to a neighbour of larger degree, so
// the parents are a transposed copy of the rows' beginnings.  Vertices of
// small degree, which cannot spare an edge, own nearly all of theirs that way;
// those of large degree are the roots where they own fewer than t units, and
// have children enough.  One pass points every vertex at its root, one pass of
// unions (a CAS on the larger root) joins the trees of a forest by arcs no
// forest holds, and vertices whose roots agree in all forests are one block.
// Vertices left outside then look for what they miss (k_pack_fill).  A round
// that unites little leaves the work to the scans, so the loop of Alg. 2 ends
// as before.
//
// What it is for: graphs whose neighbourhoods spread (k-cores of skewed
// graphs, random graphs).  There the scans' regions meet before any certifies
// much, and a round ended in the full scan, one pop after another.  Solve
// times before and after: 50-core of an R-MAT graph of scale 18 (21 K
// vertices, lambda-hat 99) 42.9 -> 0.26 ms, 10-core at scale 20 (247 K
// vertices, 14.5 M edges, lambda-hat 12) 5.05 -> 0.23 ms, two joined random
// blocks of 2048 vertices 3.13 -> 0.30 ms.  On clustered graphs (hyperbolic,
// n = 2^20) the forests fall apart into stretches that differ from forest to
// forest -- 0.4 % of the vertices united after 0.59 ms -- while the scans
// unite 95 % in 0.75 ms; the solver tells the two apart by the share of closed
// wedges (mc_graph.cu, k_graph_stats).
//
// Bound by L2 latency and random sectors: per unit of weight 8 bytes of arcs,
// one store and about eight loads of parents.
#include <algorithm>

#include "mc_internal.cuh"

namespace mc {

namespace {

constexpr int kThreads = 256;
constexpr int kReps = 8;       // blocks whose members are found by comparing roots
constexpr int kSample = 256;   // vertices the representatives come from
constexpr int kParts = 4;      // threads a sampled vertex gets
constexpr int kWideN = 65536;  // below: a warp a vertex in the starting pass

// t forests over n vertices, forest j's parent of v at F[j * n + v].  An edge
// belongs to its end of smaller degree (of equal ones, to the larger number):
// head[v] = the beginning of v's row whose owned arcs the forests started
// with; taken: a bit per arc in its owner's row, set when a forest took it
// later.
struct Pack {
    int *F;
    int *head;
    u32 *taken;
    int n, t;
};

__device__ __forceinline__ bool owns(int u, i64 du, int v, i64 dv) { return du < dv || (du == dv && u > v); }

// the 32-bit mixer "lowbias32" of C. Wellons' published hash search (2018)
__device__ __forceinline__ unsigned mix32(unsigned x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    return x ^ (x >> 16);
}

__device__ __forceinline__ int warp_incl_sum(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

__device__ __forceinline__ void add_unions(int un, Status *st) {
    un = (int)__reduce_add_sync(0xffffffffu, (unsigned)un);
    if ((threadIdx.x & 31) == 0 && un)
        atomicAdd(reinterpret_cast<unsigned long long *>(&st->unions), (unsigned long long)un);
}

// A vertex deals its units out from a forest that depends on its number (one
// for every 32 vertices): the smallest neighbours head every row and would all
// have their children in the first forests otherwise.
__device__ __forceinline__ int first_forest(int u, int t) { return (int)(mix32((unsigned)u >> 5) % (unsigned)t); }

// the rows' beginnings looked at: past them lie hubs' arcs to smaller degrees
__device__ __forceinline__ int head_limit(int a0, int a1, int t) { return a1 - a0 > 2 * t + 16 ? a0 + 2 * t + 16 : a1; }

// The starting forests, a thread a vertex: the 32 vertices of a warp fill the
// same forest at a time, so that a store is one line.  Four arcs go through at
// once, so that their neighbours' degrees are on the way together (n = 2^20,
// t = 6: 160 us one by one, 110 us so).
__global__ void __launch_bounds__(kThreads) k_pack_start(const DevGraph g, Pack P) {
    constexpr int kB = 4;
    for (int u = blockIdx.x * blockDim.x + threadIdx.x; u < g.n; u += gridDim.x * blockDim.x) {
        const int a0 = g.rp[u], a1 = head_limit(a0, g.rp[u + 1], P.t);
        const i64 du = g.deg[u];
        int i = a0, q = 0, j = first_forest(u, P.t);
        while (q < P.t && i < a1) {
            int2 e[kB];
            i64 dv[kB];
#pragma unroll
            for (int k = 0; k < kB; ++k) e[k] = i + k < a1 ? g.adj[i + k] : make_int2(u, 0);
#pragma unroll
            for (int k = 0; k < kB; ++k) dv[k] = g.deg[e[k].x];
#pragma unroll
            for (int k = 0; k < kB; ++k) {
                if (q >= P.t || i >= a1) break;
                ++i;
                if (!owns(u, du, e[k].x, dv[k])) continue;
                for (int c = e[k].y; c > 0 && q < P.t; --c, ++q) {
                    P.F[j * P.n + u] = e[k].x;
                    if (++j == P.t) j = 0;
                }
            }
        }
        P.head[u] = i - a0;
        for (; q < P.t; ++q) {
            P.F[j * P.n + u] = u;
            if (++j == P.t) j = 0;
        }
    }
}

// The same with a warp a vertex, the arcs dealt by a running sum of their
// weights, where a thread a vertex leaves the GPU idle (21 K vertices, t = 99:
// 55 us with a thread each, 24 us so; 247 K vertices, t = 12: 29 against 66).
__global__ void __launch_bounds__(kThreads) k_pack_start_wide(const DevGraph g, Pack P) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int u = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < g.n; u += nw) {
        const int a0 = g.rp[u], a1 = head_limit(a0, g.rp[u + 1], P.t);
        const i64 du = g.deg[u];
        const int j0 = first_forest(u, P.t);
        int q = 0, head = 0;
        for (int i0 = a0; i0 < a1 && q < P.t; i0 += 32) {
            const int i = i0 + lane;
            int c = 0, v = u;
            if (i < a1) {
                const int2 e = g.adj[i];
                v = e.x;
                if (owns(u, du, v, g.deg[v])) c = e.y < P.t ? e.y : P.t;
            }
            const int inc = warp_incl_sum(c), s = q + inc - c;  // s: this arc's first unit
            for (int k = s; k < s + c && k < P.t; ++k) {
                const int j = j0 + k < P.t ? j0 + k : j0 + k - P.t;
                P.F[j * P.n + u] = v;
            }
            const unsigned dealt = __ballot_sync(0xffffffffu, c > 0 && s < P.t);
            if (dealt) head = i0 - a0 + 32 - __clz(dealt);
            q += __shfl_sync(0xffffffffu, inc, 31);
        }
        for (int k = q + lane; k < P.t; k += 32) {
            const int j = j0 + k < P.t ? j0 + k : j0 + k - P.t;
            P.F[j * P.n + u] = u;
        }
        if (lane == 0) P.head[u] = head;
    }
}

// every vertex points at its root; forest after forest, so that the parents
// walked over stay in L2.  Bound by their latency (41 long-scoreboard stalls an
// issue); 21 K vertices, t = 99: 15 and 11 us, 20 and 17 on four times the blocks.
__global__ void __launch_bounds__(kFlatThreads, kFlatBlocks) k_pack_flatten(Pack P) {
    const unsigned total = (unsigned)P.n * (unsigned)P.t, stride = gridDim.x * blockDim.x;
    flatten_rounds([&](auto fresh) {
        bool any = false;
        for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += stride) {
            int *p = P.F + k / (unsigned)P.n * (unsigned)P.n;
            const int u = (int)(k % (unsigned)P.n);
            const int p0 = ld_parent(p + u), r = root_near<fresh.value>(p, p0, &any);
            if (r != p0) p[u] = r;
        }
        return any;
    });
}

// One union a vertex and forest, for every `every`-th 32 vertices of a forest
// (another 32 in the next): an owned arc behind the row's head, if it connects
// anything.  About weight / t of a vertex's units are spare, and a forest's
// trees are fewer than a tenth of its vertices, so a share of the vertices
// that falls as the rows grow joins nearly all of them.  Bound by parents from
// L2: 21 K vertices, t = 99, 31 us (52 with a walk to the root from each end).
__global__ void __launch_bounds__(kThreads) k_pack_join(const DevGraph g, Pack P, unsigned every) {
    const unsigned m = ((P.n + 31u) / 32u + every - 1u) / every * 32u, total = m * (unsigned)P.t;
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned k = blockIdx.x * blockDim.x + threadIdx.x; k < total; k += stride) {
        const unsigned j = k / m, o = k % m;
        const unsigned uu = ((o >> 5) * every + j % every) * 32u + (o & 31u);
        if (uu >= (unsigned)P.n) continue;
        const int u = (int)uu;
        const int a0 = g.rp[u] + P.head[u], len = g.rp[u + 1] - a0;
        if (len <= 0) continue;
        const i64 du = g.deg[u];
        int i = a0 + (int)(mix32(uu * 31u + j) % (unsigned)(len < 16 ? len : 16));
        int v = g.adj[i].x;
        if (!owns(u, du, v, g.deg[v])) {
            i = a0;
            v = g.adj[i].x;
            if (!owns(u, du, v, g.deg[v])) continue;
        }
        int *p = P.F + j * (unsigned)P.n;
        if (uf_meet<false>(p, u, v) != 1) continue;
        const u32 bit = 1u << (i & 31);
        if (atomicOr(&P.taken[i >> 5], bit) & bit) continue;  // another forest has it
        if (uf_meet<true>(p, u, v) != 1) atomicAnd(&P.taken[i >> 5], ~bit);
    }
}

// the vertices whose roots (by a hash of all t) are shared by most of kSample
// evenly spaced ones, most first; -1 after the last
__global__ void __launch_bounds__(kSample * kParts) k_pack_reps(Pack P, int *reps, int *giant) {
    constexpr int kH = 2 * kSample;
    __shared__ unsigned long long key[kH];
    __shared__ int cnt[kH], who[kH];
    __shared__ unsigned long long best;
    for (int i = threadIdx.x; i < kH; i += blockDim.x) {
        key[i] = ~0ULL;
        cnt[i] = 0;
        who[i] = INT_MAX;
    }
    const int u = (int)(((long long)(threadIdx.x / kParts) * P.n) / kSample);
    unsigned long long sig = 0;
#pragma unroll 4
    for (int j = threadIdx.x % kParts; j < P.t; j += kParts)
        sig += splitmix64(((u64)j << 32) | (unsigned)P.F[j * P.n + u]);
#pragma unroll
    for (int o = 1; o < kParts; o <<= 1) sig += __shfl_xor_sync(0xffffffffu, sig, o);
    sig >>= 1;  // never the empty key
    __syncthreads();
    if (threadIdx.x % kParts == 0) {
        unsigned h = (unsigned)(sig >> 20) & (kH - 1);
        while (true) {
            const unsigned long long k = atomicCAS(&key[h], ~0ULL, sig);
            if (k == ~0ULL || k == sig) break;
            h = (h + 1) & (kH - 1);
        }
        atomicAdd(&cnt[h], 1);
        atomicMin(&who[h], u);
    }
    for (int r = 0; r < kReps; ++r) {
        __syncthreads();
        if (threadIdx.x == 0) best = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < kH; i += blockDim.x)
            if (cnt[i] > 0) atomicMax(&best, ((unsigned long long)cnt[i] << 32) | (unsigned)(INT_MAX - who[i]));
        __syncthreads();
        const int v = best ? INT_MAX - (int)(best & 0xFFFFFFFFu) : -1;
        for (int i = threadIdx.x; i < kH; i += blockDim.x)
            if (who[i] == v) cnt[i] = 0;
        if (threadIdx.x == 0) {
            reps[r] = v;
            if (r == 0) *giant = v;
        }
    }
}

// the representatives' roots, kReps rows of t, in shared memory; how many
__device__ __forceinline__ int stage_reps(const Pack &P, const int *reps, int *rr) {
    int nr = 0;
    for (; nr < kReps && reps[nr] >= 0; ++nr)
        for (int j = threadIdx.x; j < P.t; j += blockDim.x) rr[nr * P.t + j] = root_of(P.F + j * P.n, reps[nr]);
    __syncthreads();
    return nr;
}

// A vertex with the same root as a representative in every forest is in its
// block: in[u] = 1 + which, 0 if none.  32 vertices a block, warp w the
// forests w, w + 8, ...
__global__ void __launch_bounds__(kThreads)
k_pack_blocks(Pack P, int *par, const int *__restrict__ reps, int *in, Status *st) {
    extern __shared__ int rr[];
    __shared__ unsigned same[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nr = stage_reps(P, reps, rr);
    int un = 0;
    for (int u0 = blockIdx.x * 32; u0 < P.n; u0 += gridDim.x * 32) {
        if (wid == 0) same[lane] = (1u << nr) - 1u;
        __syncthreads();
        const int u = u0 + lane;
        unsigned m = (1u << nr) - 1u;
        if (u < P.n) {
#pragma unroll 4
            for (int j = wid; j < P.t; j += kThreads / 32) {
                const int x = P.F[j * P.n + u];
                for (int r = 0; r < nr; ++r)
                    if (x != rr[r * P.t + j]) m &= ~(1u << r);
            }
            atomicAnd(&same[lane], m);
        }
        __syncthreads();
        if (wid == 0 && u < P.n) {
            m = same[lane];
            in[u] = __ffs(m);
            if (m && reps[__ffs(m) - 1] != u) un += uf_union(par, u, reps[__ffs(m) - 1]);
        }
        __syncthreads();
    }
    add_unions(un, st);
}

// A vertex outside the representatives' blocks looks for what it misses: the
// forests that hold it apart from the block of its first neighbour in one
// take a unit each of arcs into that block no forest holds.  With all of them
// served it is in the block.  An edge between two vertices outside is used by
// neither until one is in.  A warp a vertex, `per` (<= 32) vertices looked
// over at a time.
__global__ void __launch_bounds__(kThreads)
k_pack_fill(const DevGraph g, Pack P, int *par, const int *__restrict__ reps, int *in, int per, Status *st) {
    extern __shared__ int rr[];
    unsigned short *miss = reinterpret_cast<unsigned short *>(rr + kReps * P.t) + (threadIdx.x >> 5) * P.t;
    const int lane = threadIdx.x & 31;
    stage_reps(P, reps, rr);
    const int nw = (gridDim.x * blockDim.x) >> 5;
    int un = 0;
    for (int v0 = ((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per; v0 < g.n; v0 += nw * per) {
        const int vl = v0 + lane;
        unsigned todo = __ballot_sync(0xffffffffu, lane < per && vl < g.n && in[vl] == 0);
        while (todo) {
            const int u = v0 + __ffs(todo) - 1;
            todo &= todo - 1;
            const int a0 = g.rp[u], a1 = g.rp[u + 1], hu = P.head[u];
            const i64 du = g.deg[u];
            int k = 0, first = a0;
            for (; first < a1; first += 32) {
                const int i = first + lane;
                const int b = i < a1 ? *(volatile int *)&in[g.adj[i].x] : 0;
                const unsigned m = __ballot_sync(0xffffffffu, b != 0);
                if (m) {
                    k = __shfl_sync(0xffffffffu, b, __ffs(m) - 1);
                    break;
                }
            }
            if (k == 0) continue;
            int nm = 0;
            for (int j0 = 0; j0 < P.t; j0 += 32) {
                const int j = j0 + lane;
                const bool off = j < P.t && uf_meet<false>(P.F + j * P.n, u, rr[(k - 1) * P.t + j]) != 0;
                const unsigned m = __ballot_sync(0xffffffffu, off);
                if (off) miss[nm + __popc(m & ((1u << lane) - 1u))] = (unsigned short)j;
                nm += __popc(m);
            }
            __syncwarp();
            int got = 0;
            bool lost = false;  // a walk that was cut off united nothing
            for (int i0 = first; i0 < a1 && got < nm; i0 += 32) {
                const int i = i0 + lane;
                int c = 0, v = u;
                if (i < a1) {
                    const int2 e = g.adj[i];
                    v = e.x;
                    if (*(volatile int *)&in[v] == k) {
                        int at = -1;  // the arc in its owner's row, behind the head
                        if (owns(u, du, v, g.deg[v])) {
                            if (i - a0 >= hu) at = i;
                        } else {
                            int lo = g.rp[v] + P.head[v], hi = g.rp[v + 1] - 1;
                            while (lo <= hi) {
                                const int mid = (lo + hi) >> 1;
                                const int x = g.adj[mid].x;
                                if (x == u) {
                                    at = mid;
                                    break;
                                }
                                if (x < u) lo = mid + 1;
                                else hi = mid - 1;
                            }
                        }
                        if (at >= 0 && !((P.taken[at >> 5] >> (at & 31)) & 1u)) c = e.y < P.t ? e.y : P.t;
                    }
                }
                const int inc = warp_incl_sum(c), s = got + inc - c;
                for (int x = s; x < s + c && x < nm; ++x) lost |= uf_meet<true>(P.F + miss[x] * P.n, u, v) < 0;
                got += __shfl_sync(0xffffffffu, inc, 31);
            }
            __syncwarp();
            if (!__any_sync(0xffffffffu, lost) && got >= nm && lane == 0) {
                un += uf_union(par, u, reps[k - 1]);
                __threadfence();  // its unions are out before it counts as in the block
                *(volatile int *)&in[u] = k;
            }
        }
    }
    add_unions(un, st);
}

int blocks_for(i64 threads) {
    i64 b = (threads + kThreads - 1) / kThreads;
    const i64 cap = (i64)num_sms() * 32;
    return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

}  // namespace

// The forests lie in the contraction's key buffer, 2 ints an arc of the input.
// Only what this input needs of it counts: a buffer kept from a larger graph
// holds more, and the rounds a graph goes through must not depend on that.
bool forest_fits(const DevGraph &g, const Work &w, i64 t) {
    const i64 words = t * (i64)g.n;
    return t >= 1 && t <= kForestMaxT && words <= 2 * w.own && words < kInt32Max;
}

int forest_round(const DevGraph &g, Work &w, i64 t, cudaStream_t s) {
    Pack P;
    P.F = reinterpret_cast<int *>(w.keysA);
    P.head = w.order;
    P.taken = reinterpret_cast<u32 *>(w.valsA);
    P.n = g.n;
    P.t = (int)t;
    int *reps = reinterpret_cast<int *>(w.red);  // min_degree's pairs, free here
    const i64 words = t * (i64)g.n;
    MC_CUDA(cudaMemsetAsync(P.taken, 0, sizeof(u32) * (size_t)(g.arcs / 32 + 1), s));
    ++::mc::g_launches;
    if (g.n < kWideN) k_pack_start_wide<<<blocks_for((i64)g.n * 32), kThreads, 0, s>>>(g, P);
    else k_pack_start<<<blocks_for(g.n), kThreads, 0, s>>>(g, P);
    const int flat = std::min(blocks_for(words), num_sms() * kFlatBlocks);
    ++::mc::g_launches; k_pack_flatten<<<flat, kFlatThreads, 0, s>>>(P);
    i64 every = g.arcs / words;
    every = every < 1 ? 1 : (every > 16 ? 16 : every);
    ++::mc::g_launches; k_pack_join<<<blocks_for(words / every + 32 * t), kThreads, 0, s>>>(g, P, (unsigned)every);
    ++::mc::g_launches; k_pack_flatten<<<flat, kFlatThreads, 0, s>>>(P);
    ++::mc::g_launches; k_pack_reps<<<1, kSample * kParts, 0, s>>>(P, reps, &w.st->giant);
    const size_t smem = sizeof(int) * kReps * (size_t)t;  // at most 32 KB
    ++::mc::g_launches; k_pack_blocks<<<blocks_for((i64)g.n * 8), kThreads, smem, s>>>(P, w.par, reps, w.T, w.st);
    // as many vertices a warp as leave every warp some
    const int warps = num_sms() * 64;
    int per = g.n / warps;
    per = per < 1 ? 1 : (per > 32 ? 32 : per);
    ++::mc::g_launches;
    k_pack_fill<<<blocks_for((i64)g.n * 32 / per), kThreads, smem + 2 * (kThreads / 32) * (size_t)t, s>>>(
        g, P, w.par, reps, w.T, per, w.st);
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

}  // namespace mc
