// Connected one-phase regions of the assembled system, for gfm_get_coarse.
//
// With a density ratio of 1000 the ghost-fluid Laplacian (Sec. 3.1) couples
// a region of one phase to the rest only through its interface faces, whose
// coefficients are of the order of the heavy phase's: what a flow is made of
// (water body, air above it, drops, bubbles), and what Jacobi iterations spend
// thousands of steps on.
//
// Regions: union-find over the non-interface faces (same phase on both
// sides), linking the larger root under the smaller, so each region's root
// is its smallest cell index whatever the order of the atomic operations.
// The up-to-kMaxCoarse largest regions of at least min_size cells are counted.
#include "gfm_internal.h"

namespace gfm {

namespace {

__device__ __forceinline__ int cc_find(int *parent, int x)
{
    volatile int *P = parent;
    for (;;) {
        const int p = P[x];
        if (p == x) return x;
        const int gp = P[p];
        if (gp != p) P[x] = gp;  // path splitting: gp is an ancestor of x
        x = p;
    }
}

__device__ __forceinline__ void cc_union(int *parent, int a, int b)
{
    for (;;) {
        a = cc_find(parent, a);
        b = cc_find(parent, b);
        if (a == b) return;
        if (a < b) {
            const int t = a;
            a = b;
            b = t;
        }
        if (atomicCAS(parent + a, a, b) == a) return;
    }
}

__global__ void k_cc_init(int n, int *parent, int *csize)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    parent[i] = i;
    csize[i] = 0;
}

// Faces with both cells of the same phase (kind 0: both dry, 1: both wet).
__global__ void k_cc_hook(int F, const int32_t *__restrict__ owner, const int32_t *__restrict__ nb,
                          const int8_t *__restrict__ kind, int *parent)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= F || kind[f] > 1) return;
    cc_union(parent, owner[f], nb[f]);
}

// Region sizes, at the roots (final here).
__global__ void k_cc_count(int n, int *parent, int *csize)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    atomicAdd(csize + cc_find(parent, i), 1);
}

__global__ void k_cc_candidates(int n, const int *__restrict__ parent, const int *__restrict__ csize, int min_size,
                                int *cand, int *counters)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || parent[i] != i || csize[i] < min_size) return;
    const int k = atomicAdd(counters, 1);
    if (k < kMaxCandidates) cand[k] = i;
}

// One warp: pick the up-to-max_k largest regions (ties: smaller root first).
__global__ void k_cc_select(const int *__restrict__ csize, const int *__restrict__ cand, int *counters, int max_k,
                            int ref, Coarse *co)
{
    const int lane = threadIdx.x;
    const int nc = min(counters[0], kMaxCandidates);
    int K = 0;
    int chosen[kMaxCoarse];
    if (ref >= 0) {
        for (int k = 0; k < max_k && k < kMaxCoarse; ++k) {
            long long best = -1;  // key = size * 2^32 + (2^31 - 1 - root)
            for (int t = lane; t < nc; t += 32) {
                const int c = cand[t];
                bool taken = false;
                for (int q = 0; q < K; ++q) taken |= (chosen[q] == c);
                if (taken) continue;
                const long long key = ((long long)csize[c] << 32) | (long long)(0x7fffffff - c);
                if (key > best) best = key;
            }
            for (int off = 16; off; off >>= 1) {
                const long long o = __shfl_xor_sync(0xffffffffu, best, off);
                if (o > best) best = o;
            }
            if (best < 0) break;
            chosen[K++] = 0x7fffffff - (int)(best & 0xffffffffLL);
        }
    }
    if (lane == 0) {
        co->K = K;
        co->n_cand = counters[0];
        for (int k = 0; k < kMaxCoarse; ++k) co->sizes[k] = k < K ? csize[chosen[k]] : 0;
    }
}

// ---- batched handles: regions per tank --------------------------------------

// One warp per tank: its up-to-max_k (<= kTankCoarse) largest regions among
// the candidates whose root lies in the tank (ties: smaller root first).
__global__ void k_cc_select_tanks(const int *__restrict__ csize, const int *__restrict__ cand, int *counters,
                                  int max_k, const int32_t *__restrict__ coff, const DevParams *__restrict__ tprm,
                                  Coarse *co, TankCoarse *tco)
{
    const int t = blockIdx.x, lane = threadIdx.x;
    const int nc = min(counters[0], kMaxCandidates);
    const int lo = coff[t], hi = coff[t + 1];
    int K = 0;
    int chosen[kTankCoarse];
    if (tprm[t].ref >= 0) {
        for (int k = 0; k < max_k && k < kTankCoarse; ++k) {
            long long best = -1;  // key = size * 2^32 + (2^31 - 1 - root)
            for (int q = lane; q < nc; q += 32) {
                const int c = cand[q];
                if (c < lo || c >= hi) continue;
                bool taken = false;
                for (int j = 0; j < K; ++j) taken |= (chosen[j] == c);
                if (taken) continue;
                const long long key = ((long long)csize[c] << 32) | (long long)(0x7fffffff - c);
                if (key > best) best = key;
            }
            for (int off = 16; off; off >>= 1) {
                const long long o = __shfl_xor_sync(0xffffffffu, best, off);
                if (o > best) best = o;
            }
            if (best < 0) break;
            chosen[K++] = 0x7fffffff - (int)(best & 0xffffffffLL);
        }
    }
    if (lane == 0) {
        TankCoarse &c = tco[t];
        c.K = K;
        for (int k = 0; k < kTankCoarse; ++k) c.sizes[k] = k < K ? csize[chosen[k]] : 0;
        if (t == 0) co->n_cand = counters[0];
    }
}

inline int blocks_for(long long work, int threads) { return (int)((work + threads - 1) / threads); }

}  // namespace

cudaError_t launch_coarse(const CoarseArgs &a, cudaStream_t s)
{
    const int T = 256;
    cudaError_t e = cudaMemsetAsync(a.counters, 0, sizeof(int), s);
    if (e != cudaSuccess) return e;
    k_cc_init<<<blocks_for(a.n, T), T, 0, s>>>(a.n, a.parent, a.csize);
    k_cc_hook<<<blocks_for(a.F, T), T, 0, s>>>(a.F, a.owner, a.neighbour, a.kind, a.parent);
    k_cc_count<<<blocks_for(a.n, T), T, 0, s>>>(a.n, a.parent, a.csize);
    k_cc_candidates<<<blocks_for(a.n, T), T, 0, s>>>(a.n, a.parent, a.csize, a.min_size, a.cand, a.counters);
    if (a.T > 0)
        k_cc_select_tanks<<<a.T, 32, 0, s>>>(a.csize, a.cand, a.counters, a.max_k, a.coff, a.tprm, a.coarse, a.tco);
    else
        k_cc_select<<<1, 32, 0, s>>>(a.csize, a.cand, a.counters, a.max_k, a.ref, a.coarse);
    return cudaGetLastError();
}

}  // namespace gfm
