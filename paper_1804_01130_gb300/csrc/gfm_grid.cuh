// Grid-wide synchronisation and double-float sums shared by the persistent
// solver kernels (device only).
#pragma once

#include "gfm_internal.h"

namespace gfm {

namespace {

__device__ __forceinline__ unsigned long long gtime()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned *p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void red_release_add_u32(unsigned *p, unsigned v)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ int ld_volatile_i32(const int *p) { return *(const volatile int *)p; }

struct Grid {
    unsigned *bar;
    int *err;
    double *partials;  // [2][kMaxNR][G]
    unsigned long long budget;
    unsigned epoch;
    int G;
    int parity;
};

// FENCE: a trailing __threadfence (0.2 us), for the kernels written with it.
// Thread 0: arrive at the grid barrier and wait for the other CTAs.  Each
// poll reads the counter and the clock (a register, not a memory access);
// the error flag, a second L2 round trip, only every 16th poll.  Returns
// false on a timeout (recorded) or an error seen while waiting.
template <bool FENCE = true>
__device__ __forceinline__ bool grid_arrive_wait(Grid &g)
{
    red_release_add_u32(g.bar, 1u);
    const unsigned target = g.epoch * (unsigned)g.G;
    unsigned long long t0 = 0;
    for (unsigned k = 0;; ++k) {
        const unsigned v = ld_acquire_u32(g.bar);
        if ((int)(v - target) >= 0) break;
        const unsigned long long now = gtime();
        if (k == 0) t0 = now;
        else if (now - t0 > g.budget) {
            atomicCAS(g.err, 0, (int)GFM_ERR_TIMEOUT);
            return false;
        }
        if ((k & 15u) == 15u && ld_volatile_i32(g.err) != 0) return false;
    }
    if (FENCE) __threadfence();
    return true;
}

// Double-float accumulator: value = hi + lo, TwoSum updates (Knuth), so a
// long FP32 sum keeps ~48 bits.  Built from FP32 adds only.
struct FF {
    float hi, lo;
};

__device__ __forceinline__ void ff_add(FF &a, float x)
{
    const float s = a.hi + x;
    const float bp = s - a.hi;
    const float e = (a.hi - (s - bp)) + (x - bp);
    a.hi = s;
    a.lo += e;
}

__device__ __forceinline__ FF ff_merge(FF a, FF b)
{
    const float s = a.hi + b.hi;
    const float bp = s - a.hi;
    float e = (a.hi - (s - bp)) + (b.hi - bp);
    e += a.lo + b.lo;
    const float hi = s + e;
    return FF{hi, e - (hi - s)};
}

__device__ __forceinline__ FF ff_shfl_tree(FF v)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        FF o;
        o.hi = __shfl_xor_sync(0xffffffffu, v.hi, off);
        o.lo = __shfl_xor_sync(0xffffffffu, v.lo, off);
        v = ff_merge(v, o);
    }
    return v;
}

}  // namespace

}  // namespace gfm
