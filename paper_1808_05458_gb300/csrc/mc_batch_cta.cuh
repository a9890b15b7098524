// mc_batch_cta.cuh -- the block-per-graph batched solver (mc_batch_cta.cu).
#pragma once

#include "mc_internal.cuh"

namespace mc {

constexpr int kCtaClasses = 3;   // by the share of a SM a graph takes: all, a half, a quarter
constexpr int kCtaMaxN = 2048;
constexpr int kCtaChainN = 96;
constexpr int kCtaMaxM = 1 << 16;

// device arrays in the layout of mc_batch_min_cut.  Class c's graphs are
// order[first[c] .. first[c] + count[c]), taken through next[c]; those not
// solved here are appended to rest[*nrest ..)
struct CtaBatch {
    const long long *voff, *aoff;
    const int *rp, *col, *w;
    const int *order;
    long long *lam_out;
    u32 *bits_out;              // may be null
    const long long *bits_off;  // word offsets, may be null
    int *err_out;
    int *next, *rest, *nrest;
    int first[kCtaClasses], count[kCtaClasses];
    u64 seed;
    int pr_level;
};
// the class of a graph of n vertices and m arcs; -1: not for this solver
int batch_cta_class(int n, long long m);
// graphs the matrix's one chain may take longer for than the packing
bool batch_cta_chain(int n);
// a launch for each class that has graphs, on its stream
int batch_cta_launch(const CtaBatch &B, const cudaStream_t (&s)[kCtaClasses]);

}  // namespace mc
