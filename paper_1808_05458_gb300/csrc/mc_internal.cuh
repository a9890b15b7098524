// mc_internal.cuh -- shared declarations of the libmincut CUDA path.
//
// Device layout of a graph (one GPU, HBM resident):
//   rp   int32[n+1]   CSR row offsets
//   src  int32[arcs]  source vertex of each arc (rows are contiguous, sorted)
//   adj  int2[arcs]   {neighbour, weight} of each arc, rows sorted by neighbour
//   deg  int64[n]     weighted degree (Sec. 2.1)
// Both directions of every undirected edge are stored.  Weights are int32,
// degrees, cut values and lambda-hat are int64.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <climits>

#include <functional>
#include <string>

#include "mc.h"

namespace mc {

using i64 = long long;
using u64 = unsigned long long;
using u32 = unsigned int;

constexpr int kWarp = 32;
constexpr i64 kInt32Max = 2147483647LL;

// number of kernels launched by this host thread (reported in mc_stats)
extern thread_local long long g_launches;

// ---------------------------------------------------------------- errors --
void set_cuda_error(cudaError_t e, const char *what);
void set_error_detail(const char *msg);

#define MC_CUDA(call)                                         \
    do {                                                      \
        cudaError_t _e = (call);                              \
        if (_e != cudaSuccess) {                              \
            ::mc::set_cuda_error(_e, #call);                  \
            return MC_ECUDA;                                  \
        }                                                     \
    } while (0)

#define MC_TRY(expr)                 \
    do {                             \
        int _rc = (expr);            \
        if (_rc != MC_OK) return _rc; \
    } while (0)

// ------------------------------------------------------------- allocation --
// Device memory comes from the stream-ordered allocator (cudaMallocAsync) on
// the graph's stream; buffers live as long as their owning mc_graph.
int dev_alloc(void **p, size_t bytes, cudaStream_t s);
void test_fail_alloc_after(long long k);  // mc_test_fail_alloc_after
bool test_alloc_hook_armed();               // the hook counts allocations now
void dev_free(void *p, cudaStream_t s);

template <class T>
int dev_alloc_n(T **p, size_t n, cudaStream_t s) {
    return dev_alloc(reinterpret_cast<void **>(p), (n ? n : 1) * sizeof(T), s);
}

// ------------------------------------------------------------------ graph --
struct DevGraph {
    int n = 0;
    i64 arcs = 0;
    int *rp = nullptr;
    int *src = nullptr;
    int2 *adj = nullptr;
    i64 *deg = nullptr;
    bool sym = false;  // every arc is known to have its mirror (not for trusted input)
};

// Device-resident status block, read back once per phase.
struct Status {
    i64 lam;            // lambda-hat (atomicMin target)
    i64 unions;         // successful unions this round
    i64 scanned_arcs;   // arcs read by CAPFOREST
    i64 scanned_verts;  // vertices scanned by CAPFOREST
    i64 scans;          // scans started
    i64 blacklisted;    // pops that hit another scan's vertex
    i64 count;          // generic counter (emitted arcs, roots, ...)
    i64 count2;         // second generic counter
    i64 mindeg;         // minimum weighted degree of the current graph
    int argmin;         // smallest vertex with that degree
    int err;            // error bits (kErr*)
    u64 cursor;         // start-vertex cursor of the concurrent scans
    int scan_ids;       // scan id counter
    int best_scan;      // scan whose alpha set lambda-hat (or -1)
    int best_len;       // prefix length of that scan
    int flip;           // the side bitmap's vertex-0 bit, before canonical polarity
    // graph creation: arcs running up and down, and a missing or unequal
    // mirror, seen while the input is built (valid when it is canonical)
    i64 sym_up, sym_down;
    int sym_bad;
    int giant;           // a vertex of the block most vertices are in (forest rounds)
    int giant_share;     // how many of the 256 vertices find_giant looks at are in it
    int wedges, closed;  // wedges probed and closed (graph creation)
    i64 tests;           // triangle tests of the second and third pass
};

constexpr int kErrAsym = 1;       // asymmetric input
constexpr int kErrRange = 2;      // neighbour out of range / bad offsets
constexpr int kErrNegW = 4;       // negative weight
constexpr int kErrOverflow = 8;   // weight or degree overflow
constexpr int kErrNoProgress = 16;

// --------------------------------------------------------------- launches --
int num_sms();

// device-wide exclusive scan of int32 counts into int32 offsets (one launch
// up to 2^19 items, two beyond); *d_total receives the sum (may be nullptr).
// tmp must hold scan_tmp_words(n) ints, cleared whole once by scan_tmp_clear,
// and serve one stream; a stuck wait sets kErrNoProgress in *err.
size_t scan_tmp_words(i64 n);
int scan_tmp_clear(int *tmp, size_t words, cudaStream_t s);
int exclusive_scan_i32(const int *d_in, int *d_out, i64 n, int *d_total, int *tmp, int *err,
                       cudaStream_t s);

// LSD radix sort of (key, value) pairs on the low `bits` bits of the keys.
// Buffers A hold the input; the result ends in A or B (returned via *in_b).
// tmp must hold radix_tmp_words(n) uint32.
size_t radix_tmp_words(i64 n);
int radix_sort_pairs(u64 *keysA, int *valsA, u64 *keysB, int *valsB, i64 n, int bits,
                     u32 *tmp, int *scan_tmp, int *err, bool *in_b, cudaStream_t s);

// Contraction workspace.
constexpr int kMinDegBlocks = 1024;  // blocks of one min_degree launch at most
constexpr int kRedMinDone = 2 * kMinDegBlocks;
constexpr int kRedBestDone = 2 * kMinDegBlocks + 1;
constexpr int kRedWords = 2 * kMinDegBlocks + 2;

struct Work {
    // per-vertex (sized n0)
    int *par = nullptr;      // union-find parents
    int *root = nullptr;     // union-find roots after a flatten (labels)
    int *lab = nullptr;      // relabel map
    int *T = nullptr;        // scan owner of each vertex (0 = unvisited)
    int *order = nullptr;    // visit index inside the owning scan
    int *cnt = nullptr;      // per-vertex counts / flags
    int *orig = nullptr;     // original vertex -> current vertex
    int *scan_tmp = nullptr;
    // min_degree's per-block pairs and block counter, the best-scan search's
    // block counter (kRed* below)
    i64 *red = nullptr;
    // per-arc (sized arcs0)
    u64 *keysA = nullptr, *keysB = nullptr;
    int *valsA = nullptr, *valsB = nullptr;
    u32 *radix_tmp = nullptr;
    // per-scan records
    i64 *rec_alpha = nullptr;
    int *rec_len = nullptr;
    // fallback scan state (dense, sized n0 / arcs0)
    int *fb_r = nullptr;
    u32 *fb_pool = nullptr;
    // side bitmap of the best cut so far (original ids)
    u32 *best_side = nullptr;
    // status
    Status *st = nullptr;
    Status *h_st = nullptr;  // pinned mirror
    i64 cap_n = 0, cap_arcs = 0;
    i64 own = 0;             // what the key buffers hold in a graph made for this input alone
    i64 last_emitted = 0;    // arcs emitted by the last contraction
    // single-warp tail solver scratch (allocated on first use)
    unsigned char *tail = nullptr;
    size_t tail_bytes = 0;
    // bucket bitmaps of the block-wide full scan (allocated on first use)
    u32 *blk = nullptr;
    size_t blk_words = 0;
};

int work_alloc(Work &w, i64 n0, i64 arcs0, cudaStream_t s);
void work_free(Work &w, cudaStream_t s);
int graph_alloc(DevGraph &g, i64 n, i64 arcs, cudaStream_t s);
void graph_free(DevGraph &g, cudaStream_t s);

// read the status block back (synchronises the stream)
int status_read(Work &w, cudaStream_t s);

// the pairs of blocks a contraction emitted, n blocks (n = 0: they went into a
// graph as usual)
struct Pairs {
    const u64 *keys = nullptr;
    const int *vals = nullptr;
    i64 m = 0;
    int wb = 0, n = 0;
};

// ---------------------------------------------------------- path steps --
// Sec. 2.1 contraction of `in` by union-find blocks in w.par (roots are the
// smallest member): writes `out`, its degrees, lambda-hat update candidates
// (st->mindeg / st->argmin) and w.lab (old vertex -> new vertex).  Merged
// weights are clamped to `clamp` (> 0).  If `flatten` is false, w.lab holds
// ready labels in [0, nc) with nc given.
// `post` (may be empty) launches more work before the final status read,
// whose Status copy the caller may then use; w.last_emitted = arcs emitted.
// With `one_block` the block of st->giant holds most vertices of `in`.
int contract_graph(const DevGraph &in, DevGraph &out, Work &w, i64 clamp, bool flatten, int nc,
                   cudaStream_t s, const std::function<int()> &post = {}, bool one_block = false,
                   Pairs *pairs = nullptr);

// canonicalise raw CSR arrays (device) into `out` (drops self-loops / zero
// weights, sums parallel arcs, sorts rows); checks symmetry if asked.
// Input still arriving from the host, in chunks of whole rows: chunk k holds
// rows [row_split[k], row_split[k + 1]) and is on the device once ready[k]
// has fired; arcs is the input's arc count (known on the host).
struct StagedInput {
    int chunks = 0;
    const int *row_split = nullptr;
    cudaEvent_t *ready = nullptr;
    i64 arcs = 0;
};
int canonicalize(int n, const int *rp, const int *col, const int *w, bool check_sym,
                 DevGraph &out, Work &wk, cudaStream_t s,
                 const StagedInput *staged = nullptr);

int union_find_init(int *par, int n, cudaStream_t s);
int connected_components(const DevGraph &g, Work &w, int *ncomp, cudaStream_t s);

// minimum degree + smallest argmin into st->mindeg / st->argmin
int min_degree(const DevGraph &g, Work &w, cudaStream_t s);
// largest arc weight into st->count, rows with exactly two arcs into
// st->count2, probed wedges and how many are closed into st->wedges / closed
int graph_stats(const DevGraph &g, Work &w, cudaStream_t s);

// concurrent capped CAPFOREST (Alg. 1): unions into w.par, alpha updates
// into st->lam, owners in w.T / w.order, records in w.rec_*.
struct ScanConfig {
    int pq_fifo = 0;
    int warps = 0;         // concurrent scan warps (0 = auto)
    int budget = 0;        // touched-vertex budget per scan (0 = auto)
    u64 seed = 0;
    int round = 0;
    int start = -1;        // full scan start vertex (-1 = from seed and round)
    long long lam_hint = 0; // lambda-hat at launch (selects the queue kind)
    int visits = 1;        // scans that may scan one vertex (concurrent scans)
    int lo = 0, hi = -1;   // concurrent scans scan only vertices in [lo, hi) (hi < 0: all)
};
int capforest_parallel(const DevGraph &g, Work &w, const ScanConfig &cfg, cudaStream_t s);
// one full CAPFOREST scan (Alg. 3) from a start vertex, single warp
int capforest_full(const DevGraph &g, Work &w, const ScanConfig &cfg, cudaStream_t s);
// true when capforest_full runs the one-warp scan of a small graph (n <= 8192,
// bound <= 63, largest-key order), whose cost is a few wide scans'
bool full_scan_is_small(int n, long long cap, bool fifo);

// one round of certificates by forest packing at bound t (mc_forest.cu):
// unions into w.par, their count into st->unions, a vertex of the largest
// block into st->giant; the forests lie in w.keysA
constexpr i64 kForestMaxT = 1024;
bool forest_fits(const DevGraph &g, const Work &w, i64 t);
int forest_round(const DevGraph &g, Work &w, i64 t, cudaStream_t s);

// side bitmaps (original vertex ids, n0 bits)
int side_from_vertex(Work &w, int n0, int vertex, cudaStream_t s);
int side_from_scan(Work &w, int n0, int scan, int len, cudaStream_t s);
int side_from_component(Work &w, int n0, cudaStream_t s);  // par = CC roots
int orig_update(Work &w, int n0, cudaStream_t s);           // orig = lab[orig]

// tests lo..level; PR3/PR4 only on edges whose shorter row has <= budget arcs
// (every edge if budget < 0)
int pr_tests_budget(const DevGraph &g, Work &w, i64 lam, int lo, int level, int budget,
                    cudaStream_t s);
// PR1/PR4 on a few arcs of every row (clustered graphs; bounds below
// kTriMaxBound); unit: every weight of g is 1
constexpr i64 kTriMaxBound = 1 << 26;
int pr_triangles(const DevGraph &g, Work &w, i64 lam, bool unit, cudaStream_t s);
// a vertex of the block that most of 256 evenly spaced vertices are in ->
// st->giant, their share (of 256) -> st->giant_share; w.root from a flatten
int find_giant(Work &w, int n, cudaStream_t s);
int flatten_labels(Work &w, int n, cudaStream_t s);   // w.root[v] = root of v in w.par
int flatten_parents(Work &w, int n, cudaStream_t s);  // w.par[v] = root of v
int round_reset(Work &w, i64 lam, cudaStream_t s);    // st->lam = lam, counters = 0
int round_start(Work &w, int n, i64 lam, cudaStream_t s);  // union_find_init + round_reset
int side_canon(Work &w, int n0, cudaStream_t s);
int iota_i32(int *a, int n, cudaStream_t s);
const std::string &error_detail();

// The full scan on caller-provided state (the allocation-free entry point):
// par = union-find parents (initialised), T and r zeroed, st->lam set, a
// pool of `pool` entries each for eslot / enext, and `blk` (blk_words words)
// for the block-wide scan's bucket bitmaps; unions are applied directly.
// Picks the same kernel as capforest_full for the same graph and bound.
int capforest_full_raw(const DevGraph &g, int *par, int *T, int *order, Status *st, i64 *rec_alpha,
                       int *rec_len, int *r, int *eslot, int *enext, int pool, u32 *blk, size_t blk_words,
                       int start, cudaStream_t s);
// block-wide full scan limits: keys 0..kBlkMaxCap, at most kBlkMaxN
// vertices, whole state on chip up to kBlkOnChipBytes of shared memory
constexpr int kBlkMaxCap = 1023;
constexpr int kBlkMaxN = 1 << 20;
constexpr size_t kBlkOnChipBytes = 200 * 1024;
// words of bucket bitmaps the block-wide full scan needs off chip (0 when its
// state fits on chip)
size_t full_block_words(int n, int cap);
int flatten_raw(int *par, int *root, int *cnt, int n, cudaStream_t s);

// many graphs, one warp per graph (layout of mc_batch_min_cut, host arrays);
// shape -1 = the tuned or default configuration, kBatchDefaultShape = the
// default whatever was chosen, with the batch copied whole before the kernels
// whatever its size; *ms_out = kernel time (in chunks: with the copies of all but
// the first)
constexpr int kBatchDefaultShape = -2;
int batch_solve(int G, const long long *vtx_off, const long long *arc_off, const int *row_ptr,
                const int *col, const int *w, const mc_options &o, long long *lambdas, u32 *bitmaps,
                const long long *bitmap_word_off, int shape, double *ms_out);
int batch_shapes();
// the remaining rounds of Alg. 2 on a small graph g in one single-warp launch
// (PR1/PR2 + degree-2 rule, full capped scan, in-warp contraction per
// round); *lam = min(*lam, lambda(g)), the side recorded through w.orig
int tail_solve(const DevGraph &g, Work &w, int limit, long long *lam, u64 seed, int pr_level, int fifo,
               int n0, cudaStream_t s);
// the same on a dense matrix in shared memory (mc_dense.cu): at most kDenseN
// vertices, a bound of at most kDenseMaxLam, the largest-key order; the bound
// found into out->lam, a lower one's side into bits_out
constexpr int kDenseN = 224;
constexpr i64 kDenseMaxLam = (1 << 22) - 1;  // a column adds up below 2^30, a key's entry below 2^31
int dense_solve(const DevGraph &g, i64 lam, u64 seed, int pr_level, Status *out, u32 *bits_out, cudaStream_t s);
// the same on a contraction's emitted pairs, whose minimum degree it takes first
constexpr i64 kDensePairs = 1 << 15;  // one block reads them: 128 a thread
bool dense_takes_pairs(i64 m, i64 cap);  // m of them, weights to cap: their sums stay below 2^31
int dense_solve_pairs(const Pairs &p, i64 lam, u64 seed, int pr_level, Status *out, u32 *bits_out, cudaStream_t s);
int tail_solve_pairs(const Pairs &p, Work &w, long long *lam, u64 seed, int pr_level, int n0, cudaStream_t s);
int side_from_bits(Work &w, int n0, const u32 *bits, cudaStream_t s);  // bit v = bits[orig[v]]
void batch_set_shape(int shape);
int batch_get_shape();

// learned proposer (mc_learn.cu)
struct Proposer;
int proposer_create(Proposer **out, const float *init);
void proposer_destroy(Proposer *p);
int proposer_set(Proposer *p, const float *w);
int proposer_get(Proposer *p, float *w);
int proposer_nparams();
int proposer_forward(Proposer &p, const DevGraph &g, long long delta, cudaStream_t s);
int proposer_backward(Proposer &p, const DevGraph &g, const unsigned *bits, double *loss, cudaStream_t s);
int proposer_adam(Proposer &p, float lr, cudaStream_t s);
int proposer_grad_copy(Proposer &p, float *out);
int proposer_logits_copy(Proposer &p, int n, float *out);
int proposer_sweep(Proposer &p, const DevGraph &g, Work &w, long long *cut, int *k_out, cudaStream_t s);
// bit v = w.root[v] < k, or w.root[w.orig[v]] < k with through_orig (ranks
// of the vertices of a contracted graph)
int side_from_rank(Work &w, int n0, int k, bool through_orig, cudaStream_t s);

// label propagation sweeps on g into labels (int32[n]; uses w.cnt, w.T and
// the radix buffers as scratch)
int label_prop(const DevGraph &g, Work &w, int iters, u64 seed, int *labels, cudaStream_t s);
// labels in w.lab (arbitrary vertex ids) -> dense ids in [0, nc) by the order
// of the label values; uses w.root / w.par as scratch
int compact_labels(Work &w, int n, int *nc, cudaStream_t s);

// ---------------------------------------------------------- device bits --
__device__ __forceinline__ u64 splitmix64(u64 x) {
    x += 0x9E3779B97F4A7C15ULL;
    x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ULL;
    x = (x ^ (x >> 27)) * 0x94D049BB133111EBULL;
    return x ^ (x >> 31);
}

// Union-find with parents always below their children (link the larger root
// under the smaller), path halving on finds.  Safe under concurrency: only
// roots are linked (by CAS) and halving only shortens paths to ancestors.
__device__ __forceinline__ int uf_find(int *par, int x) {
    volatile int *p = par;
    while (true) {
        int px = p[x];
        if (px == x) return x;
        int gx = p[px];
        if (gx == px) return px;
        p[x] = gx;
        x = gx;
    }
}

// the parent of x as this SM last saw it: an older parent is an ancestor all
// the same (parents only move towards the root), so it may come from L1.  It
// should where many threads walk to one root: a million warps that fetch that
// root's word from L2 wait for its one slice (k_tri_* in
// mc_pr.cu)
__device__ __forceinline__ int ld_parent(const int *p) {
    int v;
    asm volatile("ld.global.ca.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Parents a walk goes over before it leaves the one it came to as its own: on a
// graph numbered along a path the unions of one kernel, each right by itself,
// leave chains as long as the graph, and walks to the root would take n loads
// that wait for one another.  (A path of 2^20 vertices: 0.9 ms the whole solve;
// 378 ms with walks that halve the chain as uf_find does, the walkers meeting at
// the same few words, 587 ms with the halving by compare and swap; flattening in
// three launches, the later two mostly with nothing to do, cost the small graphs
// 20 us a solve.)
constexpr int kWalk = 64;

__device__ __forceinline__ int ld_parent_l2(const int *p) {
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// the root above x, or the ancestor kWalk parents up (*far)
template <bool FRESH>
__device__ __forceinline__ int root_near(const int *p, int x, bool *far) {
    for (int k = 0; k < kWalk; ++k) {
        const int q = FRESH ? ld_parent_l2(p + x) : ld_parent(p + x);
        if (q == x) return x;
        x = q;
    }
    *far = true;
    return x;
}

// Flattens parents in rounds.  `round` walks up from all vertices of this thread
// (root_near), leaves what a walk that was cut off came to as the vertex's parent,
// and says whether there were any.  A thread writes its own vertices' parents
// alone, so that a round of all threads divides what is left of every chain by
// kWalk; the first reads through L1, the others what the rounds before wrote.  On
// grids of the resident threads at most: what lies above is not shortened before
// its thread begins.
constexpr int kFlatThreads = 256, kFlatBlocks = 8;  // a SM
template <bool V>
struct Fresh {
    static constexpr bool value = V;
};
template <class F>
__device__ __forceinline__ void flatten_rounds(F round) {
    bool more = round(Fresh<false>());
    while (more) more = round(Fresh<true>());
}

// the root above x in parents that are flat
__device__ __forceinline__ int root_of(const int *p, int x) {
    while (true) {
        const int q = ld_parent(p + x);
        if (q == x) return x;
        x = q;
    }
}

// Both ends walk up, the one with the larger parent first, until they meet or
// that one is a root: parents are smaller than their children (in a forest,
// past the first, whose parents are roots by then), so the ends are apart, and
// UNITE links the root below the other's parent.  On a chain that is a few steps
// where the ends are near each other, whatever its length.  1: apart (and
// united); 0: together; -1: neither after `most` parents.  What is read may be
// old: a root that is none any more fails its CAS (which returns its parent as
// it is), and an ancestor stays one.
constexpr int kMeet = 1024;
template <bool UNITE>
__device__ __forceinline__ int uf_meet(int *p, int a, int b, int most = kMeet) {
    int pa = ld_parent(p + a), pb = ld_parent(p + b);
    for (int k = 0; k < most; ++k) {
        if (pa == pb) return 0;
        if (pa < pb) {
            int t = a;
            a = b;
            b = t;
            t = pa;
            pa = pb;
            pb = t;
        }
        if (pa == a) {
            if (!UNITE) return 1;
            const int old = atomicCAS(p + a, a, pb);
            if (old == a) return 1;
            pa = old;
            continue;
        }
        a = pa;
        pa = ld_parent(p + a);
    }
    return -1;
}

// as uf_union; *root = the root of the merged set (its smallest member)
__device__ __forceinline__ bool uf_union_root(int *par, int a, int b, int *root) {
    while (true) {
        a = uf_find(par, a);
        b = uf_find(par, b);
        if (a == b) { *root = a; return false; }
        if (a > b) { int t = a; a = b; b = t; }
        if (atomicCAS(&par[b], b, a) == b) { *root = a; return true; }
    }
}

__device__ __forceinline__ bool uf_union(int *par, int a, int b) {
    while (true) {
        a = uf_find(par, a);
        b = uf_find(par, b);
        if (a == b) return false;
        if (a > b) { int t = a; a = b; b = t; }
        if (atomicCAS(&par[b], b, a) == b) return true;
    }
}

__device__ __forceinline__ i64 ld_volatile_i64(const i64 *p) {
    return *reinterpret_cast<const volatile i64 *>(p);
}

inline int div_up(i64 a, i64 b) { return (int)((a + b - 1) / b); }

}  // namespace mc
