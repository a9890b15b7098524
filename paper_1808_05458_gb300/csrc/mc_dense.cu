// mc_dense.cu -- the launch of the dense rounds (mc_dense.cuh) on a graph in
// device memory.
#include "mc_dense.cuh"

namespace mc {

namespace {

using DenseSmem = dense::DenseSmem<kDenseN>;
constexpr int kN = kDenseN;

__global__ void __launch_bounds__(dense::kThreads)
k_dense(DevGraph g, i64 lam0, u64 seed, int pr_level, Status *out, u32 *bits_out) {
    extern __shared__ __align__(16) unsigned char raw[];
    DenseSmem &s = *reinterpret_cast<DenseSmem *>(raw);
    int *M = s.M;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int n0 = g.n;
    if (tid == 0) s.lam = lam0;
    for (int i = tid; i < n0 * kN / 4; i += dense::kThreads) reinterpret_cast<int4 *>(M)[i] = make_int4(0, 0, 0, 0);
    for (int i = lane; i < kN; i += 32) s.acc[wid][i] = 0;
    if (tid < kN) s.deg[tid] = 0;
    s.orig[tid] = (unsigned short)tid;
    __syncthreads();
    for (int i = tid; i < (int)g.arcs; i += dense::kThreads) {
        const int2 e = g.adj[i];
        const int u = g.src[i], c = e.y < (int)lam0 ? e.y : (int)lam0;
        M[u * kN + e.x] = c;
        atomicAdd(&s.deg[u], c);
    }
    if (tid < n0) M[tid * kN + tid] = dense::kSelf;
    __syncthreads();
    const int err = dense::rounds(s, n0, seed, pr_level);
    if (s.lam < lam0 && tid < (n0 + 31) / 32) bits_out[tid] = s.best[tid];
    if (tid == 0) {
        out->lam = s.lam;
        out->err = err;
    }
}

}  // namespace

int dense_solve(const DevGraph &g, i64 lam, u64 seed, int pr_level, Status *out, u32 *bits_out, cudaStream_t s) {
    MC_CUDA(cudaFuncSetAttribute(k_dense, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(DenseSmem)));
    ++::mc::g_launches; k_dense<<<1, dense::kThreads, sizeof(DenseSmem), s>>>(g, lam, seed, pr_level, out, bits_out);
    MC_CUDA(cudaGetLastError());
    return MC_OK;
}

}  // namespace mc
