// mc_dense.cu -- the dense rounds (mc_dense.cuh) on a graph in device memory, or
// on the weights between blocks that a contraction has emitted: adding those up
// in the matrix takes the place of the sort, the sums, the rows and the minimum
// degree of a contracted graph, eight and more launches that each serve a few
// thousand pairs.  RHG 2^20, degree 32: 711 -> 597 us a solve; two blocks of
// 2048 vertices: 390 -> 311.
#include "mc_dense.cuh"

namespace mc {

namespace {

using DenseSmem = dense::DenseSmem<kDenseN>;
constexpr int kN = kDenseN;

__device__ __forceinline__ void clear(DenseSmem &s, int n0, i64 lam0) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    if (tid == 0) s.lam = lam0;
    for (int i = tid; i < n0 * kN / 4; i += dense::kThreads) reinterpret_cast<int4 *>(s.M)[i] = make_int4(0, 0, 0, 0);
    for (int i = lane; i < kN; i += 32) s.acc[wid][i] = 0;
    if (tid < kN) s.deg[tid] = 0;
    s.orig[tid] = (unsigned short)tid;
    __syncthreads();
}

__device__ __forceinline__ void finish(DenseSmem &s, int n0, i64 lam0, u64 seed, int pr_level, Status *out,
                                       u32 *bits_out) {
    const int err = dense::rounds(s, n0, seed, pr_level);
    if (s.lam < lam0 && (int)threadIdx.x < (n0 + 31) / 32) bits_out[threadIdx.x] = s.best[threadIdx.x];
    if (threadIdx.x == 0) {
        out->lam = s.lam;
        out->err = err;
    }
}

__global__ void __launch_bounds__(dense::kThreads)
k_dense(DevGraph g, i64 lam0, u64 seed, int pr_level, Status *out, u32 *bits_out) {
    extern __shared__ __align__(16) unsigned char raw[];
    DenseSmem &s = *reinterpret_cast<DenseSmem *>(raw);
    int *M = s.M;
    const int tid = threadIdx.x;
    const int n0 = g.n;
    clear(s, n0, lam0);
    for (int i = tid; i < (int)g.arcs; i += dense::kThreads) {
        const int2 e = g.adj[i];
        const int u = g.src[i], c = e.y < (int)lam0 ? e.y : (int)lam0;
        M[u * kN + e.x] = c;
        atomicAdd(&s.deg[u], c);
    }
    if (tid < n0) M[tid * kN + tid] = dense::kSelf;
    __syncthreads();
    finish(s, n0, lam0, seed, pr_level, out, bits_out);
}

// m pairs of blocks (key a * n0 + b, in both directions) with their weights, in
// the low wb bits of the key or, without (wb = 0), in vals
__global__ void __launch_bounds__(dense::kThreads)
k_dense_pairs(const u64 *__restrict__ keys, const int *__restrict__ vals, int m, int wb, int n0, i64 lam0, u64 seed,
              int pr_level, Status *out, u32 *bits_out) {
    extern __shared__ __align__(16) unsigned char raw[];
    DenseSmem &s = *reinterpret_cast<DenseSmem *>(raw);
    int *M = s.M;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    clear(s, n0, lam0);
#pragma unroll 4
    for (int i = tid; i < m; i += dense::kThreads) {
        const u64 k = keys[i];
        const unsigned key = (unsigned)(k >> wb);
        const int c = wb ? (int)(k & ((1ull << wb) - 1ull)) : vals[i];
        const unsigned a = key / (unsigned)n0, b = key % (unsigned)n0;
        atomicAdd(&M[a * kN + b], c);
    }
    __syncthreads();
    for (int a = wid; a < n0; a += dense::kWarps) {
        int d = 0;
        for (int b = lane; b < n0; b += 32) {
            int c = M[a * kN + b];
            c = c < (int)lam0 ? c : (int)lam0;
            M[a * kN + b] = b == a ? dense::kSelf : c;
            d += c;
        }
        d = (int)__reduce_add_sync(dense::kAll, (unsigned)d);
        if (lane == 0) s.deg[a] = d;
    }
    __syncthreads();
    dense::take_min_degree(s, n0, n0);
    finish(s, n0, lam0, seed, pr_level, out, bits_out);
}

}  // namespace

int dense_solve(const DevGraph &g, i64 lam, u64 seed, int pr_level, Status *out, u32 *bits_out, cudaStream_t s) {
    MC_CUDA(cudaFuncSetAttribute(k_dense, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DenseSmem)));
    ++::mc::g_launches; k_dense<<<1, dense::kThreads, sizeof(DenseSmem), s>>>(g, lam, seed, pr_level, out, bits_out);
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

bool dense_takes_pairs(i64 m, i64 cap) { return m <= kDensePairs && m * cap <= INT_MAX; }

int dense_solve_pairs(const Pairs &p, i64 lam, u64 seed, int pr_level, Status *out, u32 *bits_out, cudaStream_t s) {
    MC_CUDA(cudaFuncSetAttribute(k_dense_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DenseSmem)));
    ++::mc::g_launches;
    k_dense_pairs<<<1, dense::kThreads, sizeof(DenseSmem), s>>>(p.keys, p.vals, (int)p.m, p.wb, p.n, lam, seed,
                                                                pr_level, out, bits_out);
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

}  // namespace mc
