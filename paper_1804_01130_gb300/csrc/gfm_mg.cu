// Multigrid-preconditioned conjugate gradients for the pinned GFM pressure
// system (Sec. 3.1; the paper names no solver), one persistent cooperative
// kernel per solve, for one mesh or a batch of tanks.
//
// Preconditioner: one symmetric V-cycle over the aggregates of
// gfm_mg_setup.cpp.  On each level two damped Jacobi sweeps before and after
// the coarse correction, with the two weights of the degree-2 Chebyshev
// polynomial on [0.35, 2] (the spectrum of D^{-1} A is in [0, 2]) in mirrored
// order, piecewise constant transfers, and the coarse operator formed by
// every assembly from the assembled face coefficients (k_mg_level).  The
// iteration count hardly depends on the mesh size: 22-52 V-cycles for a
// relative residual of 1e-12 on tanks up to 20 times as long as deep, where
// Jacobi iterations number 184 to 6600.  On longer, shallower tanks the merged
// cells mix water and air: up to 315 V-cycles (529x13 cells, 120 depths long).
//
// A V-cycle on the mesh level is five passes over the rows (two sweeps, the
// residual, two sweeps), all of them gathers of ONE vector, against the one
// pass of a Jacobi iteration; the coarse levels add a third (2D) or a
// seventh (3D).  The FP32 operator is applied in difference form, sum_f
// gamma_f (x_i - x_j) + pin_i x_i, which keeps the zero row sums of the GFM
// Laplacian exact; the FP64 one in diagonal form.  The CG direction needs no pass of its own gathers: s = A p is updated as
// s = A z + beta s.
//
// Precision.  GFM_FP64 (T = double): everything FP64; the result is accepted
// on the true residual b - A x, from which the directions start anew.  The
// steps are summed in e and folded into x there, so that x carries one
// rounding and not one per step: where the rounding of x is all that is left of
// the residual this is 5-10% less, as low as the Jacobi form gets.  GFM_MIXED (T = float): FP32 iterations with
// double-float dot products inside FP64 residual replacement, as the Jacobi
// forms: when the FP32 residual has dropped by three decades (or claims
// convergence) e is folded into x in FP64 and r becomes the true FP64
// residual; the direction is kept.  Replacing after four decades instead of
// three was slower everywhere: FP32 residuals that far down cost more
// iterations than the replacements saved (256x128x128 box 12.5 against
// 10.3 ms, 1024x512 tank 3.36 against 3.20 ms, 64 tanks 24.4 against 22.8 ms).
//
// Levels too small to share between CTAs run in CTA 0 alone, in its shared
// memory, while the others wait at the grid barrier (from MgArgs::tail on).
//
// Batches: rows of all tanks form one block-diagonal system, so the V-cycle
// needs no tank bookkeeping; only the dot products, alpha, beta and the
// stopping tests are per tank.  CTAs own equal contiguous stretches of slices
// across tank borders; a CTA writes one partial sum per (CTA, tank) segment,
// to slot CTA + tank, and every CTA adds each tank's segments in the same
// order, so all CTAs take identical decisions and results are
// bit-reproducible.  A tank that has converged, or waits for the others to ask
// for a replacement, gives its share of the CTAs to those still iterating.
#include "gfm_grid.cuh"

namespace gfm {

namespace {

constexpr int kMgNR = 2;       // most values one all-reduce sums
constexpr float kOm1 = 0.56418f;  // Chebyshev degree 2 on [0.35, 2]: 1 / (1.175 +- 0.825 cos(pi/4))
constexpr float kOm2 = 1.69016f;
constexpr int kSegLane = 8;    // tanks with more segments are summed by a warp
// Most iterations between residual replacements, after which the stall test
// ends a solve that gets nowhere.  FP64: far above what a solve takes (20 to
// 240), since every replacement restarts its directions.
constexpr int kMgCheck32 = 40, kMgCheck64 = 400;
// A residual claims convergence at a tenth of the tolerance (squared here).
// What a V-cycle leaves of it is smoother than what Jacobi iterations leave, and
// p_d's error the larger for the same residual: at 0.9 of the tolerance it
// exceeded the Jacobi form's in a quarter of 151 tanks (solves, steps, adjoints of
// 800 to 150,000 cells), at 0.3 in 12%, at 0.1 in 6%, there by rounding; the times
// are 1 : 1.024 : 1.048, the mean errors 1 : 0.39 : 0.20.
constexpr double kMgClaim = 0.01;

enum MgAct : int { kMgGo = 0, kMgConverged = 1, kMgNotConverged = 2, kMgBreakdown = 3 };
enum MgFlag : int { kFlagNone = 0, kFlagUpdate = 1, kFlagRestart = 2, kFlagCap = 3 };

struct MgShared {
    double2 warp_p[32][kMgNR];   // partial sums of the warps (double, or a double-float pair)
    double bnorm[kMaxTanks], sc[kMaxTanks], isc[kMaxTanks], gam[kMaxTanks], rho_max[kMaxTanks], rho[kMaxTanks];
    double best[kMaxTanks], rho_stop[kMaxTanks], xavg[kMaxTanks];
    double tot[kMgNR][kMaxTanks];
    float al32[kMaxTanks], be32[kMaxTanks];
    double al64[kMaxTanks], be64[kMaxTanks];
    int act[kMaxTanks], flag[kMaxTanks], wait[kMaxTanks], fresh[kMaxTanks];
    int iters[kMaxTanks], updates[kMaxTanks], stall[kMaxTanks], last_rep[kMaxTanks], restarts[kMaxTanks];
    int c0[kMaxTanks], c1[kMaxTanks];  // first and last CTA holding slices of the tank
    int seg_s0[kMaxTanks], seg_s1[kMaxTanks], seg_tank[kMaxTanks];  // this CTA's segments
    int wide[kMaxTanks];
    int nseg, n_wide, any_active, any_flag, replan, fail, polish;
};

// ---- sums ------------------------------------------------------------------
// Accumulators: double-float for the FP32 iterations' dot products, double otherwise.
__device__ __forceinline__ void acc_add(FF &a, float x) { ff_add(a, x); }
__device__ __forceinline__ void acc_add(double &a, double x) { a += x; }
__device__ __forceinline__ FF acc_merge(FF a, FF b) { return ff_merge(a, b); }
__device__ __forceinline__ double acc_merge(double a, double b) { return a + b; }
__device__ __forceinline__ FF acc_shfl(FF v, int off)
{
    return FF{__shfl_xor_sync(0xffffffffu, v.hi, off), __shfl_xor_sync(0xffffffffu, v.lo, off)};
}
__device__ __forceinline__ double acc_shfl(double v, int off) { return __shfl_xor_sync(0xffffffffu, v, off); }
__device__ __forceinline__ double acc_value(FF v) { return (double)v.hi + (double)v.lo; }
__device__ __forceinline__ double acc_value(double v) { return v; }
template <typename A>
__device__ __forceinline__ A acc_tree(A v)
{
#pragma unroll
    for (int off = 16; off; off >>= 1) v = acc_merge(v, acc_shfl(v, off));
    return v;
}
template <typename T>
struct AccOf {
    using type = double;
};
template <>
struct AccOf<float> {
    using type = FF;
};

struct Ctx {
    Grid g;
    MgShared *sh;
    int T, lane, warp, nw;
    int P;  // partial slots per value (grid + tanks)
};

// Plain grid barrier (an error raised elsewhere is seen at the next wait).
// Thread 0's acquire and the CTA barrier order the other CTAs' writes before
// every thread's reads; a V-cycle passes some twenty of these.
__device__ __forceinline__ bool mg_sync(Ctx &c)
{
    __syncthreads();
    c.g.epoch += 1u;
    if (threadIdx.x == 0) c.sh->fail = grid_arrive_wait<false>(c.g) ? 0 : 1;
    __syncthreads();
    return c.sh->fail == 0;
}

// Sum the CTA's per-thread values of one segment and write them to its slot.
template <int NR, typename A>
__device__ __forceinline__ void put_partials(Ctx &c, int tank, const A (&v)[NR])
{
    MgShared &sh = *c.sh;
    A r[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) r[k] = acc_tree(v[k]);
    __syncthreads();
    if (c.lane == 0) {
#pragma unroll
        for (int k = 0; k < NR; ++k) *reinterpret_cast<A *>(&sh.warp_p[c.warp][k]) = r[k];
    }
    __syncthreads();
    if (c.warp == 0) {
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            A t = c.lane < c.nw ? *reinterpret_cast<const A *>(&sh.warp_p[c.lane][k]) : A{};
            t = acc_tree(t);
            if (c.lane == 0)
                reinterpret_cast<A *>(c.g.partials)[((size_t)c.g.parity * kMgNR + k) * c.P + blockIdx.x + tank] = t;
        }
    }
}

// After every segment's put_partials: grid barrier, then sh.tot[k][t] = the
// sum of value k over tank t's segments, the same bits in every CTA.
template <int NR, typename A>
__device__ __forceinline__ bool mg_allreduce(Ctx &c)
{
    MgShared &sh = *c.sh;
    if (!mg_sync(c)) return false;
    const A *src = reinterpret_cast<const A *>(c.g.partials) + (size_t)c.g.parity * kMgNR * c.P;
    auto get = [&](int k, int slot) {
        if constexpr (sizeof(A) == sizeof(float2)) {
            const float2 t = __ldcg(reinterpret_cast<const float2 *>(src + (size_t)k * c.P + slot));
            A a;
            memcpy(&a, &t, sizeof a);
            return a;
        }
    };
    if (sh.n_wide < c.T)
        for (int q = threadIdx.x; q < NR * c.T; q += blockDim.x) {
            const int k = q / c.T, t = q - k * c.T;
            const int n = sh.c1[t] - sh.c0[t] + 1;
            if (n > kSegLane) continue;
            A v[kSegLane];
#pragma unroll
            for (int j = 0; j < kSegLane; ++j) v[j] = j < n ? get(k, sh.c0[t] + j + t) : A{};
            sh.tot[k][t] = acc_value(acc_merge(acc_merge(acc_merge(v[0], v[1]), acc_merge(v[2], v[3])),
                                               acc_merge(acc_merge(v[4], v[5]), acc_merge(v[6], v[7]))));
        }
    for (int q = c.warp; q < NR * sh.n_wide; q += c.nw) {
        const int k = q / sh.n_wide, t = sh.wide[q - k * sh.n_wide];
        A v[6];  // 192 segments with every load in flight
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            const int b = sh.c0[t] + c.lane + 32 * j;
            v[j] = b <= sh.c1[t] ? get(k, b + t) : A{};
        }
        A acc = acc_merge(acc_merge(acc_merge(v[0], v[1]), acc_merge(v[2], v[3])), acc_merge(v[4], v[5]));
        for (int b = sh.c0[t] + c.lane + 192; b <= sh.c1[t]; b += 32) acc = acc_merge(acc, get(k, b + t));
        acc = acc_tree(acc);
        if (c.lane == 0) sh.tot[k][t] = acc_value(acc);
    }
    c.g.parity ^= 1;
    __syncthreads();
    return true;
}

// ---- row passes --------------------------------------------------------------
// The rows' off-diagonal parts, in the form each precision can afford:
//  float:  acc_i = sum_k val (x_i - x_j), which keeps the zero row sums exact
//          under FP32 rounding; A x = acc + pin x.
//  double: acc_i = sum_k val x_j, half the instructions of the FP64 pipe
//          (64 cycles each per quarter SM); A x = diag x - acc, and a sweep
//          x + w D^{-1} (b - A x) = (1 - w) x + w D^{-1} (b + acc).
template <typename T>
__device__ __forceinline__ T row_add(T acc, T g, T xi, T xj)
{
    if constexpr (sizeof(T) == 8) return fma(g, xj, acc);
    else return fma(g, xi - xj, acc);
}
// A x of a row; p its pin (float) or diagonal (double)
template <typename T>
__device__ __forceinline__ T row_ax(T acc, T x, T p)
{
    if constexpr (sizeof(T) == 8) return fma(p, x, -acc);
    else return fma(p, x, acc);
}
// x + w d (b - A x)
template <typename T>
__device__ __forceinline__ T row_sweep(T acc, T x, T b, T w, T d, T p)
{
    if constexpr (sizeof(T) == 8) return fma(w * d, b + acc, (T(1) - w) * x);
    else return fma(w * d, b - fma(p, x, acc), x);
}

// This CTA's share of the mesh's table in shared memory (col == nullptr: not
// held): slice pointers and slots from slice s0, slot base on.
template <typename T>
struct RowCache {
    const int32_t *sp, *col;
    const T *val;
    int s0, base;
};

// Rows of slices s0 + w0, + nw, ... below s1 (U of them in flight per warp,
// chunks of CH faces), then op.post(i, x_i, acc_i, pre) with pre = op.pre(i)
// loaded before the gathers.
template <typename T, int CH, int U, bool FINE, typename Op>
__device__ __forceinline__ void row_pass(const MgLevel &lv, const RowCache<T> &rc, const T *X, int s0, int s1, int w0,
                                         int nw, int lane, int n, Op &op)
{
    const bool held = FINE && rc.col != nullptr;
    const T *__restrict__ val = static_cast<const T *>(lv.val);
    const int32_t *__restrict__ col = lv.col;
    for (int sb = s0 + w0; sb < s1; sb += U * nw) {
        int base[U], w[U];
        T xi[U], acc[U];
        typename Op::Pre pr[U];
        int wmax = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = sb + u * nw, i = s * kSlice + lane;
            base[u] = 0;
            w[u] = 0;
            xi[u] = T(0);
            acc[u] = T(0);
            if (s < s1 && i < n) {
                if (held) {
                    base[u] = rc.sp[s - rc.s0];
                    w[u] = (rc.sp[s - rc.s0 + 1] - base[u]) >> 5;
                } else {
                    base[u] = __ldg(lv.sp + s);
                    w[u] = (__ldg(lv.sp + s + 1) - base[u]) >> 5;
                }
                xi[u] = X[i];
                pr[u] = op.pre(i);
            }
            wmax = max(wmax, w[u]);
        }
        for (int k0 = 0; k0 < wmax; k0 += CH) {
            int j[U][CH];
            T gm[U][CH], xj[U][CH];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < CH; ++q) {
                    const bool ok = k0 + q < w[u];
                    const int slot = base[u] + (k0 + q) * kSlice + lane;
                    if (FINE && held) {
                        j[u][q] = ok ? rc.col[slot - rc.base] : 0;
                        gm[u][q] = ok ? rc.val[slot - rc.base] : T(0);
                    } else if constexpr (FINE) {  // read once per pass
                        j[u][q] = ok ? __ldcs(col + slot) : 0;
                        gm[u][q] = ok ? __ldcs(val + slot) : T(0);
                    } else {
                        j[u][q] = ok ? __ldg(col + slot) : 0;
                        gm[u][q] = ok ? __ldg(val + slot) : T(0);
                    }
                }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < CH; ++q) xj[u][q] = (k0 + q < w[u]) ? X[j[u][q]] : xi[u];
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int q = 0; q < CH; ++q) acc[u] = row_add(acc[u], gm[u][q], xi[u], xj[u][q]);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int s = sb + u * nw, i = s * kSlice + lane;
            if (s < s1 && i < n) op.post(i, xi[u], acc[u], pr[u]);
        }
    }
}

// What a row needs of its diagonal: the pin (float; on the mesh one cell of
// the tank, on a coarse level an array that is zero but for the aggregate
// holding the pinned cell), or the diagonal (double, an array).
template <typename T, bool FINE>
struct Pin {
    const T *a;
    int ref;
    T pin;
    __device__ __forceinline__ T at(int i) const
    {
        if constexpr (FINE && sizeof(T) == 4) return i == ref ? pin : T(0);
        else return a[i];
    }
};

// out = x + w D^{-1} (b - A x)
template <typename T, bool FINE>
struct SweepOp {
    struct Pre {
        T b, d, p;
    };
    const T *b, *dinv;
    T *out;
    T w;
    Pin<T, FINE> pin;
    __device__ __forceinline__ Pre pre(int i) const
    {
        return Pre{b[i], dinv[i], sizeof(T) == 8 ? T(0) : pin.at(i)};
    }
    __device__ __forceinline__ void post(int i, T x, T acc, const Pre &p)
    {
        out[i] = row_sweep(acc, x, p.b, w, p.d, p.p);
    }
};

// out = b - A x
template <typename T, bool FINE>
struct ResidOp {
    struct Pre {
        T b, p;
    };
    const T *b;
    T *out;
    Pin<T, FINE> pin;
    __device__ __forceinline__ Pre pre(int i) const { return Pre{b[i], pin.at(i)}; }
    __device__ __forceinline__ void post(int i, T x, T acc, const Pre &p) { out[i] = p.b - row_ax(acc, x, p.p); }
};

// The last sweep on the mesh: z = x + w D^{-1} (r - A x), and r.z.
template <typename T>
struct LastOp {
    struct Pre {
        T b, d, p;
    };
    const T *b, *dinv;
    T *out;
    T w;
    Pin<T, true> pin;
    typename AccOf<T>::type sum;
    __device__ __forceinline__ Pre pre(int i) const
    {
        return Pre{b[i], dinv[i], sizeof(T) == 8 ? T(0) : pin.at(i)};
    }
    __device__ __forceinline__ void post(int i, T x, T acc, const Pre &p)
    {
        const T z = row_sweep(acc, x, p.b, w, p.d, p.p);
        out[i] = z;
        acc_add(sum, p.b * z);
    }
};

// fine[child] += z for the children of node i of a level.
template <typename T>
__device__ __forceinline__ void add_to_children(const MgLevel &lv, T *fine, int i, T z)
{
    const int s = i >> 5, lane = i & 31;
    const int c0 = __ldg(lv.cp + s), w0 = (__ldg(lv.cp + s + 1) - c0) >> 5;
    for (int k = 0; k < w0; k += 4) {
        int ch[4];
        T v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) ch[q] = k + q < w0 ? __ldg(lv.child + c0 + (k + q) * kSlice + lane) : -1;
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = ch[q] >= 0 ? fine[ch[q]] : T(0);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (ch[q] >= 0) fine[ch[q]] = v[q] + z;
    }
}

// The last sweep on a coarse level, its result added to the children.
template <typename T>
struct LastCoarseOp {
    struct Pre {
        T b, d, p;
    };
    const MgLevel &lv;
    T *fine;
    T w;
    Pin<T, false> pin;
    __device__ __forceinline__ Pre pre(int i) const
    {
        return Pre{static_cast<const T *>(lv.b)[i], static_cast<const T *>(lv.dinv)[i],
                   sizeof(T) == 8 ? T(0) : pin.at(i)};
    }
    __device__ __forceinline__ void post(int i, T x, T acc, const Pre &p)
    {
        add_to_children<T>(lv, fine, i, row_sweep(acc, x, p.b, w, p.d, p.p));
    }
};

// s = A z + beta s, p = z + beta p (fresh: s = A z, p = z), and p.s.
template <typename T>
struct DirOp {
    struct Pre {
        T p, s, pin;
    };
    T *P, *S;
    T be;
    bool fresh;
    Pin<T, true> pin;
    typename AccOf<T>::type sum;
    __device__ __forceinline__ Pre pre(int i) const
    {
        return fresh ? Pre{T(0), T(0), pin.at(i)} : Pre{P[i], S[i], pin.at(i)};
    }
    __device__ __forceinline__ void post(int i, T x, T acc, const Pre &p)
    {
        const T s = fma(be, p.s, row_ax(acc, x, p.pin));
        const T d = fma(be, p.p, x);
        S[i] = s;
        P[i] = d;
        acc_add(sum, d * s);
    }
};

// b = the sum of the children's residuals, x = w D^{-1} b (the first sweep from zero).
template <typename T>
__device__ __forceinline__ void restrict_pass(const MgLevel &lv, const T *res, T w, int s0, int s1, int w0, int nw,
                                              int lane)
{
    const T *dinv = static_cast<const T *>(lv.dinv);
    T *b = static_cast<T *>(lv.b), *x = static_cast<T *>(lv.xa);
    for (int s = s0 + w0; s < s1; s += nw) {
        const int i = s * kSlice + lane;
        const int c0 = __ldg(lv.cp + s), cw = (__ldg(lv.cp + s + 1) - c0) >> 5;
        const T d = i < lv.n ? dinv[i] : T(0);
        T sum = T(0);
        for (int k = 0; k < cw; k += 4) {
            int ch[4];
            T v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) ch[q] = k + q < cw ? __ldg(lv.child + c0 + (k + q) * kSlice + lane) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = ch[q] >= 0 ? res[ch[q]] : T(0);
            sum += (v[0] + v[1]) + (v[2] + v[3]);
        }
        if (i < lv.n) {
            b[i] = sum;
            x[i] = w * d * sum;
        }
    }
}

__device__ __forceinline__ void split(int ns, int G, int b, int &s0, int &s1)
{
    s0 = (int)(((long long)ns * b) / G);
    s1 = (int)(((long long)ns * (b + 1)) / G);
}

// ---- the tail: small levels in CTA 0's shared memory -------------------------
template <int N>
struct Int {
    static constexpr int value = N;
};

// Barrier t + 1 over the first `nwarps` warps (one warp: a warp barrier).
__device__ __forceinline__ void tail_bar(int t, int nwarps)
{
    if (nwarps == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(t + 1), "r"(nwarps * 32) : "memory");
}

// Stage the tail levels' tables (constant during a solve), all threads of CTA 0.
// Padding slots point at the row itself with coefficient 0; a missing child at
// the element after the finer vector's last, which xa keeps at 0.
template <typename T>
__device__ void tail_stage(const MgArgs &a, unsigned char *dsm)
{
    for (int l = a.tail; l < a.L; ++l) {
        const MgTail &q = a.tl[l - a.tail];
        const MgLevel &lv = a.lv[l];
        T *val = reinterpret_cast<T *>(dsm + q.val), *dinv = reinterpret_cast<T *>(dsm + q.dinv);
        T *pin = reinterpret_cast<T *>(dsm + q.pin), *xa = reinterpret_cast<T *>(dsm + q.xa);
        uint16_t *col = reinterpret_cast<uint16_t *>(dsm + q.col), *child = reinterpret_cast<uint16_t *>(dsm + q.child);
        int32_t *gchild = reinterpret_cast<int32_t *>(dsm + q.child);
        if (threadIdx.x == 0) xa[q.np] = T(0);
        for (int i = threadIdx.x; i < q.np; i += blockDim.x) {
            const bool on = i < q.n;
            dinv[i] = on ? static_cast<const T *>(lv.dinv)[i] : T(0);
            pin[i] = on ? static_cast<const T *>(lv.pin)[i] : T(0);
            const int s = i >> 5, lane = i & 31;
            const int base = __ldg(lv.sp + s), w = (__ldg(lv.sp + s + 1) - base) >> 5;
            for (int k = 0; k < q.w; ++k) {
                const int slot = base + k * kSlice + lane;
                val[k * q.np + i] = k < w ? __ldg(static_cast<const T *>(lv.val) + slot) : T(0);
                col[k * q.np + i] = (uint16_t)(k < w ? __ldg(lv.col + slot) : i);
            }
            const int c0 = __ldg(lv.cp + s), cw = (__ldg(lv.cp + s + 1) - c0) >> 5;
            for (int k = 0; k < q.cw; ++k) {
                const int ch = k < cw ? __ldg(lv.child + c0 + k * kSlice + lane) : -1;
                if (l == a.tail) gchild[k * q.np + i] = ch;
                else child[k * q.np + i] = (uint16_t)(ch >= 0 ? ch : a.tl[l - a.tail - 1].np);
            }
        }
    }
    __syncthreads();
}

// The rows a thread holds of one tail level, W faces each (padded), in registers.
template <typename T, int W, int R>
struct TailRows {
    T val[R][W], d[R], pin[R];
    int col[R][W];
    __device__ __forceinline__ TailRows(const MgTail &q, const unsigned char *dsm, int tid, int nth)
    {
        const T *v = reinterpret_cast<const T *>(dsm + q.val);
        const uint16_t *cl = reinterpret_cast<const uint16_t *>(dsm + q.col);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = tid + r * nth;
            const bool on = r == 0 || i < q.np;
#pragma unroll
            for (int k = 0; k < W; ++k) {
                const bool ok = on && k < q.w;
                val[r][k] = ok ? v[k * q.np + i] : T(0);
                col[r][k] = ok ? (int)cl[k * q.np + i] : 0;
            }
            d[r] = on ? reinterpret_cast<const T *>(dsm + q.dinv)[i] : T(0);
            pin[r] = on ? reinterpret_cast<const T *>(dsm + q.pin)[i] : T(0);
        }
    }
    __device__ __forceinline__ T off_diagonal(int r, T xi, const T *x) const
    {
        T xj[W], acc = T(0);
#pragma unroll
        for (int k = 0; k < W; ++k) xj[k] = x[col[r][k]];
#pragma unroll
        for (int k = 0; k < W; ++k) acc = row_add(acc, val[r][k], xi, xj[k]);
        return acc;
    }
    // b - A x of row r, xi its own value; and a sweep with weight w
    __device__ __forceinline__ T resid(int r, T b, T xi, const T *x) const
    {
        return b - row_ax(off_diagonal(r, xi, x), xi, pin[r]);
    }
    __device__ __forceinline__ T sweep(int r, T b, T xi, T w, const T *x) const
    {
        return row_sweep(off_diagonal(r, xi, x), xi, b, w, d[r], pin[r]);
    }
};

// One tail level of the V-cycle on the way down (restriction, two sweeps,
// residual into xa) and on the way up (two sweeps, the result added to the
// children).  t = 0: the children are in global memory.
template <typename T, int W, int R>
__device__ __forceinline__ void tail_down(const MgArgs &a, unsigned char *dsm, int t, bool last, int nwp)
{
    const MgTail &q = a.tl[t];
    const int nth = nwp * 32, tid = threadIdx.x;
    const T om1 = T(kOm1), om2 = T(kOm2);
    auto vec = [&](int off) { return reinterpret_cast<T *>(dsm + off); };
    T *b = vec(q.b), *xa = vec(q.xa), *xb = vec(q.xb);
    T br[R], x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) br[r] = T(0);
    if (t == 0) {
        const T *res = static_cast<const T *>(a.lv[a.tail - 1].res);
        const int32_t *child = reinterpret_cast<const int32_t *>(dsm + q.child);
        for (int k = 0; k < q.cw; k += 4) {
            T v[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = tid + r * nth;
                    const int ch = (i < q.np && k + u < q.cw) ? child[(k + u) * q.np + i] : -1;
                    v[r][u] = ch >= 0 ? res[ch] : T(0);
                }
#pragma unroll
            for (int r = 0; r < R; ++r) br[r] += (v[r][0] + v[r][1]) + (v[r][2] + v[r][3]);
        }
    } else {
        const T *res = vec(a.tl[t - 1].xa);
        const uint16_t *child = reinterpret_cast<const uint16_t *>(dsm + q.child);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = tid + r * nth;
            if (i < q.np)
                for (int k = 0; k < q.cw; ++k) br[r] += res[child[k * q.np + i]];
        }
    }
    const TailRows<T, W, R> row(q, dsm, tid, nth);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * nth;
        x[r] = om1 * row.d[r] * br[r];
        if (i < q.np) {
            b[i] = br[r];
            xa[i] = x[r];
        }
    }
    tail_bar(t, nwp);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * nth;
        x[r] = row.sweep(r, br[r], x[r], om2, xa);
        if (i < q.np) xb[i] = x[r];
    }
    tail_bar(t, nwp);
    if (last) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * nth;
        const T v = row.resid(r, br[r], x[r], xb);
        if (i < q.np) xa[i] = v;
    }
    tail_bar(t, nwp);
}

template <typename T, int W, int R>
__device__ __forceinline__ void tail_up(const MgArgs &a, unsigned char *dsm, int t, bool last, int nwp)
{
    const MgTail &q = a.tl[t];
    const int nth = nwp * 32, tid = threadIdx.x;
    const T om1 = T(kOm1), om2 = T(kOm2);
    auto vec = [&](int off) { return reinterpret_cast<T *>(dsm + off); };
    T *xa = vec(q.xa), *xb = vec(q.xb);
    T br[R], x[R];
    const TailRows<T, W, R> row(q, dsm, tid, nth);
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * nth;
        br[r] = i < q.np ? vec(q.b)[i] : T(0);
    }
    if (!last) tail_bar(t, nwp);  // the coarser level's correction is in xb
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = tid + r * nth;
        x[r] = i < q.np ? xb[i] : T(0);
        x[r] = row.sweep(r, br[r], x[r], om2, xb);
        if (i < q.np) xa[i] = x[r];
    }
    tail_bar(t, nwp);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = row.sweep(r, br[r], x[r], om1, xa);
    if (t == 0) {
        T *fine = static_cast<T *>(a.lv[a.tail - 1].xb);
        const int32_t *child = reinterpret_cast<const int32_t *>(dsm + q.child);
        for (int k = 0; k < q.cw; k += 4) {
            int ch[R][4];
            T v[R][4];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int i = tid + r * nth;
                    ch[r][u] = (i < q.np && k + u < q.cw) ? child[(k + u) * q.np + i] : -1;
                    v[r][u] = ch[r][u] >= 0 ? fine[ch[r][u]] : T(0);
                }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (ch[r][u] >= 0) fine[ch[r][u]] = v[r][u] + x[r];
        }
    } else {
        T *fine = vec(a.tl[t - 1].xb);
        const uint16_t *child = reinterpret_cast<const uint16_t *>(dsm + q.child);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = tid + r * nth;
            if (i < q.np)
                for (int k = 0; k < q.cw; ++k) fine[child[k * q.np + i]] += x[r];
        }
    }
}

// Rows per thread and faces per row of a level, as template arguments (the
// plan admits two rows a thread up to six faces, else one, up to kMgTailWidth
// faces).
template <typename T, bool UP>
__device__ __forceinline__ void tail_level(const MgArgs &a, unsigned char *dsm, int t, bool last, int nwp)
{
    auto go = [&](auto w, auto r) {
        if constexpr (UP) tail_up<T, decltype(w)::value, decltype(r)::value>(a, dsm, t, last, nwp);
        else tail_down<T, decltype(w)::value, decltype(r)::value>(a, dsm, t, last, nwp);
    };
    const int w = a.tl[t].w;
    if (a.tl[t].np > nwp * 32) {
        if (w <= 4) go(Int<4>{}, Int<2>{});
        else go(Int<6>{}, Int<2>{});
    } else {
        if (w <= 4) go(Int<4>{}, Int<1>{});
        else if (w <= 6) go(Int<6>{}, Int<1>{});
        else go(Int<kMgTailWidth>{}, Int<1>{});
    }
}

// The V-cycle over the tail levels, from the residual of level tail - 1 to the
// correction added to its xb.  Level t is worked on by the first ceil(n / 32)
// warps and closed by its own named barrier, so the last levels cost a warp
// barrier per pass.  What it costs is a chain of short passes (five a level):
// each keeps its rows in registers and touches only shared memory.  For the
// 2048-node level of the 1024x512 tank and the five below it: 32 us when the
// passes read global memory, 19 us now, the two grid barriers and the first
// level's transfers (about 7 us) included.
template <typename T>
__device__ void tail_cycle(const MgArgs &a, const Ctx &c, unsigned char *dsm)
{
    const int nt = a.L - a.tail;
    auto warps = [&](int t) { return min(c.nw, a.tl[t].np >> 5); };
    int t = 0;
    for (; t < nt && c.warp < warps(t); ++t) tail_level<T, false>(a, dsm, t, t + 1 == nt, warps(t));
    for (--t; t >= 0; --t) tail_level<T, true>(a, dsm, t, t + 1 == nt, warps(t));
}

// A row pass on a coarse level (two slices in flight per warp measured the same).
template <typename T, int CH, typename Op>
__device__ __forceinline__ void coarse_pass(const MgLevel &lv, const T *X, int s0, int s1, const Ctx &c, Op &op)
{
    row_pass<T, CH, 1, false>(lv, RowCache<T>{}, X, s0, s1, c.warp, c.nw, c.lane, lv.n, op);
}

// Levels 1 .. L-1 of the V-cycle, from the mesh's residual (lv[0].res) to the
// correction added to lv[0].xb.  Ends with a grid barrier.
template <typename T, int CH>
__device__ __forceinline__ bool coarse_cycle(const MgArgs &a, Ctx &c, unsigned char *dsm)
{
    const int L = a.L;
    const T om1 = T(kOm1), om2 = T(kOm2);
    int s0, s1;
    for (int l = 1; l < a.tail; ++l) {
        const MgLevel &lv = a.lv[l];
        const Pin<T, false> pin{static_cast<const T *>(lv.pin), -1, T(0)};
        split(lv.n_slices, c.g.G, blockIdx.x, s0, s1);
        restrict_pass<T>(lv, static_cast<const T *>(a.lv[l - 1].res), om1, s0, s1, c.warp, c.nw, c.lane);
        if (!mg_sync(c)) return false;
        SweepOp<T, false> sw{static_cast<const T *>(lv.b), static_cast<const T *>(lv.dinv), static_cast<T *>(lv.xb), om2, pin};
        coarse_pass<T, CH>(lv, static_cast<const T *>(lv.xa), s0, s1, c, sw);
        if (!mg_sync(c)) return false;
        if (l + 1 < L) {
            ResidOp<T, false> rs{static_cast<const T *>(lv.b), static_cast<T *>(lv.res), pin};
            coarse_pass<T, CH>(lv, static_cast<const T *>(lv.xb), s0, s1, c, rs);
            if (!mg_sync(c)) return false;
        }
    }
    if (a.tail < L) {
        if (blockIdx.x == 0) tail_cycle<T>(a, c, dsm);
        if (!mg_sync(c)) return false;
    }
    for (int l = a.tail - 1; l >= 1; --l) {
        const MgLevel &lv = a.lv[l];
        const Pin<T, false> pin{static_cast<const T *>(lv.pin), -1, T(0)};
        split(lv.n_slices, c.g.G, blockIdx.x, s0, s1);
        SweepOp<T, false> sw{static_cast<const T *>(lv.b), static_cast<const T *>(lv.dinv), static_cast<T *>(lv.xa), om2, pin};
        coarse_pass<T, CH>(lv, static_cast<const T *>(lv.xb), s0, s1, c, sw);
        if (!mg_sync(c)) return false;
        LastCoarseOp<T> lc{lv, static_cast<T *>(a.lv[l - 1].xb), om1, pin};
        coarse_pass<T, CH>(lv, static_cast<const T *>(lv.xa), s0, s1, c, lc);
        if (!mg_sync(c)) return false;
    }
    return true;
}

// (A x)_i in FP64, difference form with the pin.
template <int CH>
__device__ __forceinline__ double row64(const SolveArgs &a, int s, int lane, double xi, double pin_i)
{
    const int base = __ldg(a.m.slice_ptr + s), w = (__ldg(a.m.slice_ptr + s + 1) - base) >> 5;
    double acc = pin_i * xi;
    for (int k0 = 0; k0 < w; k0 += CH) {
        int j[CH];
        double gm[CH], xj[CH];
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            const bool ok = k0 + q < w;
            const int slot = base + (k0 + q) * kSlice + lane;
            j[q] = ok ? __ldcs(a.m.col + slot) : 0;
            gm[q] = ok ? __ldcs(a.m.val64 + slot) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < CH; ++q) xj[q] = (k0 + q < w) ? a.x64[j[q]] : xi;
#pragma unroll
        for (int q = 0; q < CH; ++q) acc = fma(gm[q], xi - xj[q], acc);
    }
    return acc;
}

__device__ void mg_abort(const MgArgs &a)
{
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int e = ld_volatile_i32(a.s.err);
        for (int t = 0; t < a.T; ++t) {
            a.s.info[t].status = e;
            a.s.info[t].rel_res_l2 = -1.0;
            a.s.info[t].rel_res_l1 = -1.0;
        }
    }
}

}  // namespace

template <typename T, int CH, int NT, int U>
__global__ void __launch_bounds__(NT, 1) k_solve_mg(MgArgs a)
{
    constexpr bool kMixed = sizeof(T) == 4;
    constexpr int UB = kMixed ? 4 : 2;  // slices in flight per warp in the update pass (U: in the row passes)
    using A = typename AccOf<T>::type;
    __shared__ MgShared sh;
    extern __shared__ __align__(16) unsigned char dsm[];
    Ctx c;
    c.g = Grid{a.s.bar, a.s.err, a.s.partials, a.s.budget_ns, 0u, (int)gridDim.x, 0};
    c.sh = &sh;
    c.T = a.T;
    c.lane = threadIdx.x & 31;
    c.warp = threadIdx.x >> 5;
    c.nw = blockDim.x >> 5;
    c.P = (int)gridDim.x + a.T;
    const int T_ = a.T, lane = c.lane, warp = c.warp, nw = c.nw;
    const T om1 = T(kOm1), om2 = T(kOm2);
    auto working = [&](int t) { return sh.act[t] == kMgGo && sh.wait[t] == 0; };
    // Share the slices of the tanks for which want(t) holds among the CTAs:
    // equal contiguous stretches across tank borders.  A pure function of the
    // tanks' state, so every CTA builds the same table.
    auto plan = [&](auto want) {
        __syncthreads();
        if (threadIdx.x < 32) {  // lane l takes tanks l, l + 32, ...
            auto first = [&](int t) { return T_ > 1 ? a.tank_off[t] >> 5 : 0; };
            auto count = [&](int t) { return (T_ > 1 ? a.tank_off[t + 1] >> 5 : a.s.m.n_slices) - first(t); };
            int ns = 0;
            for (int t = lane; t < T_; t += 32) ns += want(t) ? count(t) : 0;
#pragma unroll
            for (int o = 16; o; o >>= 1) ns += __shfl_xor_sync(0xffffffffu, ns, o);
            // with the mesh's table held in shared memory, CTA 0 has the tail's there
            const int skip = a.cache_slots > 0 && a.tail < a.L ? 1 : 0;
            const long long G = min(c.g.G - skip, ns), b = (long long)blockIdx.x - skip, N = max(ns, 1);
            const bool on = b >= 0 && b < G;
            const int lo = on ? (int)(N * b / G) : ns, hi = on ? (int)(N * (b + 1) / G) : ns;
            int off0 = 0, m = 0, nwd = 0;
            for (int t0 = 0; t0 < T_; t0 += 32) {
                const int t = t0 + lane;
                const int n = t < T_ && want(t) ? count(t) : 0;
                int inc = n;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, inc, o);
                    if (lane >= o) inc += y;
                }
                const int off = off0 + inc - n;
                int c0 = 0, c1 = -1;
                if (n > 0) {
                    c0 = (int)(((off + 1) * G - 1) / N) + skip;
                    c1 = (int)(((off + n) * G - 1) / N) + skip;
                }
                if (t < T_) {
                    sh.c0[t] = c0;
                    sh.c1[t] = c1;
                }
                const unsigned below = (1u << lane) - 1u;
                const bool wide = c1 - c0 + 1 > kSegLane, here = n > 0 && off < hi && off + n > lo;
                const unsigned wm = __ballot_sync(0xffffffffu, wide), hm = __ballot_sync(0xffffffffu, here);
                if (wide) sh.wide[nwd + __popc(wm & below)] = t;
                if (here) {
                    const int q = m + __popc(hm & below);
                    sh.seg_s0[q] = first(t) + max(off, lo) - off;
                    sh.seg_s1[q] = first(t) + min(off + n, hi) - off;
                    sh.seg_tank[q] = t;
                }
                m += __popc(hm);
                nwd += __popc(wm);
                off0 += __shfl_sync(0xffffffffu, inc, 31);
            }
            if (lane == 0) {
                sh.nseg = m;
                sh.n_wide = nwd;
            }
        }
        __syncthreads();
    };
    plan([](int) { return true; });
    if (blockIdx.x == 0 && a.tail < a.L) tail_stage<T>(a, dsm);
    // Hold this CTA's share of the mesh's table in shared memory where every
    // CTA's fits (a single mesh, whose shares stay the same): the passes then
    // wait for one L2 round trip per row, the gathers', instead of three.
    // 1024x512 cells in FP32, us a pass: 9.4 -> 6.6.
    RowCache<T> rc{};
    if (a.cache_slots > 0 && sh.nseg > 0) {
        const int s0 = sh.seg_s0[0], ns = sh.seg_s1[0] - s0, base = a.s.m.slice_ptr[s0];
        int32_t *sp = reinterpret_cast<int32_t *>(dsm), *col = sp + a.cache_slices + 1;
        T *val = reinterpret_cast<T *>(dsm + a.cache_val);
        for (int k = threadIdx.x; k <= ns; k += blockDim.x) sp[k] = a.s.m.slice_ptr[s0 + k];
        const int total = a.s.m.slice_ptr[s0 + ns] - base;
        for (int k = threadIdx.x; k < total; k += blockDim.x) {
            col[k] = a.s.m.col[base + k];
            val[k] = static_cast<const T *>(a.lv[0].val)[base + k];
        }
        rc = RowCache<T>{sp, col, val, s0, base};
        __syncthreads();
    }
    auto bail = [&]() { mg_abort(a); };

    const MgLevel &l0 = a.lv[0];
    T *R = static_cast<T *>(l0.b), *XA = static_cast<T *>(l0.xa), *XB = static_cast<T *>(l0.xb);
    T *RES = static_cast<T *>(l0.res), *Z = static_cast<T *>(a.z), *P = static_cast<T *>(a.p), *S = static_cast<T *>(a.sv);
    T *E = static_cast<T *>(a.e);  // correction since the last replacement
    const T *dinv = static_cast<const T *>(l0.dinv);
    // pinned cell and end of the real cells of a tank
    auto tank_end = [&](int t) { return T_ > 1 ? a.tank_off[t] + a.s.n_per_tank[t] : a.s.m.n; };
    auto tank_pin = [&](int t) {
        const DevParams *p = T_ > 1 ? a.tprm + t : a.s.prm;
        return Pin<T, true>{static_cast<const T *>(l0.pin), p->ref, T(p->pin64)};
    };

    // prologue: x0, ||b||
    for (int q = 0; q < sh.nseg; ++q) {
        const int t = sh.seg_tank[q], end = tank_end(t);
        double vb[1] = {0.0};
        for (int s = sh.seg_s0[q] + warp; s < sh.seg_s1[q]; s += nw) {
            const int i = s * kSlice + lane;
            if (i < end) {
                a.s.x64[i] = a.s.use_x0 ? a.s.p_user[a.s.iperm[i]] : 0.0;
                E[i] = T(0);
                const double bi = a.s.b[i];
                vb[0] = fma(bi, bi, vb[0]);
            }
        }
        put_partials<1, double>(c, t, vb);
    }
    if (!mg_allreduce<1, double>(c)) { bail(); return; }
    for (int t = threadIdx.x; t < T_; t += blockDim.x) {
        const double bb = sh.tot[0][t], bn = bb > 0.0 ? sqrt(bb) : 1.0;
        sh.bnorm[t] = bn;
        int ex = 0;
        // FP32: one power-of-two scale for the whole solve, so residual
        // entries start near 1 and shrink by at most the tolerance
        if constexpr (kMixed) frexp(bn / sqrt((double)(a.s.n_per_tank ? a.s.n_per_tank[t] : a.s.m.n)), &ex);
        sh.sc[t] = ldexp(1.0, -ex);
        sh.isc[t] = ldexp(1.0, ex);
        sh.rho_stop[t] = (a.s.rtol * bn * sh.sc[t]) * (a.s.rtol * bn * sh.sc[t]);
        sh.gam[t] = 1.0;
        sh.rho[t] = 0.0;
        sh.act[t] = kMgGo;
        sh.flag[t] = kFlagRestart;  // the first residual, no direction yet
        sh.wait[t] = 0;
        sh.fresh[t] = 1;
        sh.iters[t] = sh.updates[t] = sh.stall[t] = sh.last_rep[t] = sh.restarts[t] = 0;
        sh.best[t] = 1e300;
    }
    __syncthreads();
    const int cap_updates = a.s.max_refine + 1 + (kMixed ? (int)(2.0 * log10(1.0 / a.s.rtol)) : 0);

    // r = b - A x (FP64) for the flagged tanks, x += e first; also
    // the V-cycle's first sweep from zero.  Then the tanks' decisions.
    // polish > 0: x += D^{-1} r on every second cell instead.  A claim refuted
    // by less than 1.4 leaves r to the rounding of x, which these sweeps undo
    // where it is largest: six of them take 15-20% off, and what the Jacobi
    // form can reach, which ends in such single-cell steps, is reached.
    auto replace_pass = [&](bool first, int polish) -> bool {
        if (T_ > 1 && !first) plan([&](int t) { return sh.flag[t] != kFlagNone; });
        if (!first) {
            for (int q = 0; q < sh.nseg; ++q) {
                const int t = sh.seg_tank[q], end = tank_end(t);
                if (sh.flag[t] == kFlagNone) continue;
                const double isc = sh.isc[t];
                for (int sb = sh.seg_s0[q] + warp; sb < sh.seg_s1[q]; sb += 4 * nw) {
                    T e[4];
                    double x[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = (sb + u * nw) * kSlice + lane;
                        const bool ok = sb + u * nw < sh.seg_s1[q] && i < end;
                        if (polish > 0) e[u] = ok && ((i ^ polish) & 1) ? dinv[i] * R[i] : T(0);
                        else e[u] = ok ? E[i] : T(0);
                        x[u] = ok ? a.s.x64[i] : 0.0;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int i = (sb + u * nw) * kSlice + lane;
                        if (sb + u * nw < sh.seg_s1[q] && i < end) {
                            a.s.x64[i] = fma((double)e[u], isc, x[u]);
                            E[i] = T(0);
                        }
                    }
                }
            }
            if (!mg_sync(c)) return false;
        }
        for (int q = 0; q < sh.nseg; ++q) {
            const int t = sh.seg_tank[q], end = tank_end(t);
            A v[1] = {A{}};
            if (sh.flag[t] != kFlagNone) {
                const double sc = sh.sc[t];
                const DevParams *pp = T_ > 1 ? a.tprm + t : a.s.prm;
                const int ref = pp->ref;
                const double pin = pp->pin64;
                const bool with_x = !first || a.s.use_x0;
                for (int s = sh.seg_s0[q] + warp; s < sh.seg_s1[q]; s += nw) {
                    const int i = s * kSlice + lane;
                    if (i < end) {
                        const double bi = a.s.b[i];
                        const T d = dinv[i];
                        const double r = with_x ? bi - row64<CH>(a.s, s, lane, a.s.x64[i], i == ref ? pin : 0.0) : bi;
                        const T rt = (T)(r * sc);
                        R[i] = rt;
                        XA[i] = om1 * d * rt;
                        acc_add(v[0], rt * rt);
                    }
                }
            }
            put_partials<1, A>(c, t, v);
        }
        if (!mg_allreduce<1, A>(c)) return false;
        if (threadIdx.x < 32) {
            bool active = false, again = false;
            for (int t = threadIdx.x; t < T_; t += 32) {
                const int f = sh.flag[t];
                if (sh.act[t] == kMgGo && f != kFlagNone) {
                    const double rr = sh.tot[0][t];
                    const double rel2 = rr / (sh.bnorm[t] * sh.sc[t] * (sh.bnorm[t] * sh.sc[t]));
                    // FP32 residual entries carry 6e-8 each: stay below the target by as much
                    const double tol2 = a.s.rtol * a.s.rtol * (kMixed ? 1.0 - 1e-6 : 1.0);
                    // the recurrence claimed half the tolerance or less, the truth is just above it
                    if (f == kFlagUpdate && polish < 6 && sh.rho[t] <= 0.25 * sh.rho_stop[t] && rel2 > tol2 &&
                        rel2 <= 2.0 * tol2) {
                        again = active = true;
                        continue;
                    }
                    sh.flag[t] = kFlagNone;
                    sh.wait[t] = 0;
                    sh.last_rep[t] = sh.iters[t];
                    ++sh.updates[t];
                    sh.fresh[t] |= (f == kFlagRestart) ? 1 : 0;
                    // the recurrence had drifted from the true residual: its
                    // direction is no longer conjugate to anything.  In FP64
                    // that holds at every replacement: one comes when the
                    // recurrence claims convergence, where the true residual
                    // may be as long as the recurrence's but is mostly the
                    // rounding of x and points elsewhere.  Steps with an old
                    // direction and a new residual made it grow there (from
                    // 6e-13 to 3e-10 and on to the iteration cap).
                    if (!kMixed || !(rr <= 4.0 * sh.rho[t])) sh.fresh[t] = 1;
                    sh.rho_max[t] = rr;
                    if (rel2 <= tol2) sh.act[t] = kMgConverged;
                    else if (f == kFlagCap) sh.act[t] = kMgNotConverged;
                    else if (!isfinite(rr)) sh.act[t] = kMgBreakdown;
                    else if (!first) {
                        if (f == kFlagRestart && ++sh.restarts[t] > 3) sh.act[t] = kMgBreakdown;
                        if (rel2 < 0.25 * sh.best[t]) {
                            sh.best[t] = rel2;
                            sh.stall[t] = 0;
                        } else {
                            ++sh.stall[t];
                        }
                        if (sh.act[t] == kMgGo && (sh.stall[t] > (kMixed ? 8 : 3) || sh.updates[t] > cap_updates))
                            sh.act[t] = kMgNotConverged;
                    } else {
                        sh.best[t] = rel2;
                        if (a.s.max_iters <= 0) sh.act[t] = kMgNotConverged;
                    }
                }
                active |= sh.act[t] == kMgGo;
            }
            active = __any_sync(0xffffffffu, active);
            again = __any_sync(0xffffffffu, again);
            if (threadIdx.x == 0) {
                sh.any_active = active;
                sh.polish = again;
            }
        }
        __syncthreads();
        if (T_ > 1) plan(working);
        return true;
    };
    auto replace = [&](bool first) -> bool {
        if (!replace_pass(first, 0)) return false;
        for (int k = 1; sh.polish; ++k)
            if (!replace_pass(false, k)) return false;
        return true;
    };
    if (!replace(true)) { bail(); return; }

    auto fine_sweep = [&](const T *X, T *out, T w) {
        for (int q = 0; q < sh.nseg; ++q) {
            const int t = sh.seg_tank[q];
            if (!working(t)) continue;
            SweepOp<T, true> op{R, dinv, out, w, tank_pin(t)};
            row_pass<T, CH, U, true>(l0, rc, X, sh.seg_s0[q], sh.seg_s1[q], warp, nw, lane, tank_end(t), op);
        }
    };
    while (sh.any_active) {
        // z = V-cycle(r): XA holds the first sweep
        fine_sweep(XA, XB, om2);
        if (!mg_sync(c)) { bail(); return; }
        if (a.L > 1) {
            for (int q = 0; q < sh.nseg; ++q) {
                const int t = sh.seg_tank[q];
                if (!working(t)) continue;
                ResidOp<T, true> op{R, RES, tank_pin(t)};
                row_pass<T, CH, U, true>(l0, rc, XB, sh.seg_s0[q], sh.seg_s1[q], warp, nw, lane, tank_end(t), op);
            }
            if (!mg_sync(c)) { bail(); return; }
            if (!coarse_cycle<T, CH>(a, c, dsm)) { bail(); return; }
        }
        fine_sweep(XB, XA, om2);
        if (!mg_sync(c)) { bail(); return; }
        for (int q = 0; q < sh.nseg; ++q) {
            const int t = sh.seg_tank[q];
            A v[1] = {A{}};
            if (working(t)) {
                LastOp<T> op{R, dinv, Z, om1, tank_pin(t), A{}};
                row_pass<T, CH, U, true>(l0, rc, XA, sh.seg_s0[q], sh.seg_s1[q], warp, nw, lane, tank_end(t), op);
                v[0] = op.sum;
            }
            put_partials<1, A>(c, t, v);
        }
        if (!mg_allreduce<1, A>(c)) { bail(); return; }
        for (int t = threadIdx.x; t < T_; t += blockDim.x) {
            if (!working(t)) continue;
            const double gn = sh.tot[0][t];
            const bool ok = gn > 0.0 && isfinite(gn);
            if (!ok) sh.flag[t] = kFlagRestart;
            const bool fresh = sh.fresh[t] || !ok;
            if constexpr (kMixed) sh.be32[t] = fresh ? 0.0f : (float)gn / (float)sh.gam[t];
            else sh.be64[t] = fresh ? 0.0 : gn / sh.gam[t];
            sh.fresh[t] = fresh;
            sh.gam[t] = gn;
        }
        __syncthreads();
        // p = z + beta p, s = A p, p.s
        for (int q = 0; q < sh.nseg; ++q) {
            const int t = sh.seg_tank[q];
            A v[1] = {A{}};
            if (working(t) && sh.flag[t] == kFlagNone) {
                T be;
                if constexpr (kMixed) be = sh.be32[t];
                else be = sh.be64[t];
                DirOp<T> op{P, S, be, sh.fresh[t] != 0, tank_pin(t), A{}};
                row_pass<T, CH, U, true>(l0, rc, Z, sh.seg_s0[q], sh.seg_s1[q], warp, nw, lane, tank_end(t), op);
                v[0] = op.sum;
            }
            put_partials<1, A>(c, t, v);
        }
        if (!mg_allreduce<1, A>(c)) { bail(); return; }
        for (int t = threadIdx.x; t < T_; t += blockDim.x) {
            if (!working(t) || sh.flag[t] != kFlagNone) continue;
            const double ps = sh.tot[0][t];
            const bool ok = ps > 0.0 && isfinite(ps);
            if constexpr (kMixed) sh.al32[t] = ok ? (float)sh.gam[t] / (float)ps : 0.0f;
            else sh.al64[t] = ok ? sh.gam[t] / ps : 0.0;
            if (!ok) sh.flag[t] = kFlagRestart;
            sh.fresh[t] = 0;
        }
        __syncthreads();
        // e += alpha p, r -= alpha s, the next V-cycle's first sweep, r.r
        for (int q = 0; q < sh.nseg; ++q) {
            const int t = sh.seg_tank[q], end = tank_end(t), e1 = sh.seg_s1[q];
            A v[1] = {A{}};
            if (working(t) && sh.flag[t] == kFlagNone) {
                T al;
                if constexpr (kMixed) al = sh.al32[t];
                else al = sh.al64[t];
                for (int sb = sh.seg_s0[q] + warp; sb < e1; sb += UB * nw) {
                    T p[UB], s[UB], r[UB], x[UB], d[UB];
#pragma unroll
                    for (int u = 0; u < UB; ++u) {
                        const int i = (sb + u * nw) * kSlice + lane;
                        const bool ok = sb + u * nw < e1 && i < end;
                        p[u] = ok ? P[i] : T(0);
                        s[u] = ok ? S[i] : T(0);
                        r[u] = ok ? R[i] : T(0);
                        x[u] = ok ? E[i] : T(0);
                        d[u] = ok ? dinv[i] : T(0);
                    }
#pragma unroll
                    for (int u = 0; u < UB; ++u) {
                        const int i = (sb + u * nw) * kSlice + lane;
                        if (sb + u * nw < e1 && i < end) {
                            E[i] = fma(al, p[u], x[u]);
                            const T rn = fma(-al, s[u], r[u]);
                            R[i] = rn;
                            XA[i] = om1 * d[u] * rn;
                            acc_add(v[0], rn * rn);
                        }
                    }
                }
            }
            put_partials<1, A>(c, t, v);
        }
        if (!mg_allreduce<1, A>(c)) { bail(); return; }
        // A tank asks for a residual replacement when its residual claims
        // convergence, can no longer be trusted in FP32 (three decades below
        // the last true one), has gone kMgCheck32 or kMgCheck64 iterations
        // without one, or cannot go on.  In a batch a tank that claims
        // convergence idles until the round, which comes when no tank is left
        // iterating or some tank must not wait.  In FP64 each claim that the
        // true residual refuted halves the next one's target: near the
        // rounding floor the true residual is the recurrence's and x's
        // rounding added up.
        if (threadIdx.x < 32) {
            bool now = false, asked = false, going = false, waits = false;
            for (int t = threadIdx.x; t < T_; t += 32) {
                if (sh.act[t] != kMgGo) continue;
                if (sh.wait[t]) {
                    asked = true;
                    continue;
                }
                if (sh.flag[t] == kFlagRestart) {
                    now = true;
                    continue;
                }
                const int it = ++sh.iters[t];
                const double rho = sh.tot[0][t];
                sh.rho[t] = rho;
                if (it >= a.s.max_iters) {
                    sh.flag[t] = kFlagCap;
                    now = true;
                } else if (!(rho > (kMixed ? kMgClaim : ldexp(kMgClaim, -2 * min(sh.updates[t] - 1, 8))) * sh.rho_stop[t])) {
                    sh.flag[t] = kFlagUpdate;
                    sh.wait[t] = 1;
                    asked = waits = true;
                } else if ((kMixed && rho <= 1e-6 * sh.rho_max[t]) ||
                           it - sh.last_rep[t] >= (kMixed ? kMgCheck32 : kMgCheck64)) {
                    sh.flag[t] = kFlagUpdate;
                    sh.wait[t] = 1;
                    asked = waits = true;
                } else {
                    going = true;
                }
            }
            now = __any_sync(0xffffffffu, now);
            asked = __any_sync(0xffffffffu, asked);
            going = __any_sync(0xffffffffu, going);
            waits = __any_sync(0xffffffffu, waits);
            if (threadIdx.x == 0) {
                sh.any_flag = now || (asked && !going);
                sh.replan = waits;
            }
        }
        __syncthreads();
        if (sh.any_flag) {
            if (!replace(false)) { bail(); return; }
        } else if (T_ > 1 && sh.replan) {
            plan(working);
        }
    }

    // the record: true FP64 residual (r in r64), solution in caller order,
    // normalised L1 residual sum|r| / (sum|A x - x_avg rowsum| + sum|b - x_avg rowsum|)
    if (T_ > 1) plan([](int) { return true; });
    if (!mg_sync(c)) { bail(); return; }
    for (int q = 0; q < sh.nseg; ++q) {
        const int t = sh.seg_tank[q], end = tank_end(t);
        const DevParams *pp = T_ > 1 ? a.tprm + t : a.s.prm;
        const int ref = pp->ref;
        const double pin = pp->pin64;
        double v[2] = {0.0, 0.0};
        for (int s = sh.seg_s0[q] + warp; s < sh.seg_s1[q]; s += nw) {
            const int i = s * kSlice + lane;
            if (i < end) {
                const double xi = a.s.x64[i];
                const double r = a.s.b[i] - row64<CH>(a.s, s, lane, xi, i == ref ? pin : 0.0);
                a.s.r64[i] = r;
                a.s.p_user[a.s.iperm[i]] = xi;
                v[0] = fma(r, r, v[0]);
                v[1] += xi;
            }
        }
        put_partials<2, double>(c, t, v);
    }
    if (!mg_allreduce<2, double>(c)) { bail(); return; }
    for (int t = threadIdx.x; t < T_; t += blockDim.x) {
        sh.xavg[t] = sh.tot[1][t] / (double)(a.s.n_per_tank ? a.s.n_per_tank[t] : a.s.m.n);
        sh.rho[t] = sh.tot[0][t];
    }
    __syncthreads();
    for (int q = 0; q < sh.nseg; ++q) {
        const int t = sh.seg_tank[q], end = tank_end(t);
        const DevParams *pp = T_ > 1 ? a.tprm + t : a.s.prm;
        const int ref = pp->ref;
        const double pin = pp->pin64, xavg = sh.xavg[t];
        double v[2] = {0.0, 0.0};
        for (int s = sh.seg_s0[q] + warp; s < sh.seg_s1[q]; s += nw) {
            const int i = s * kSlice + lane;
            if (i < end) {
                const double r = a.s.r64[i], bi = a.s.b[i], rs = i == ref ? pin : 0.0;
                v[0] += fabs(r);
                v[1] += fabs(bi - r - xavg * rs) + fabs(bi - xavg * rs);
            }
        }
        put_partials<2, double>(c, t, v);
    }
    if (!mg_allreduce<2, double>(c)) { bail(); return; }
    if (blockIdx.x == 0)
        for (int t = threadIdx.x; t < T_; t += blockDim.x) {
            const int e = ld_volatile_i32(a.s.err);
            int st = GFM_OK;
            if (sh.act[t] == kMgNotConverged) st = GFM_ERR_NOT_CONVERGED;
            else if (sh.act[t] == kMgBreakdown) st = GFM_ERR_BREAKDOWN;
            if (e != 0) st = e;
            a.s.info[t].iters = sh.iters[t];
            a.s.info[t].refinements = sh.updates[t];
            a.s.info[t].status = st;
            a.s.info[t].reserved = 0;
            a.s.info[t].rel_res_l2 = sqrt(sh.rho[t]) / sh.bnorm[t];
            a.s.info[t].rel_res_l1 = sh.tot[0][t] / (sh.tot[1][t] + 1e-300);
        }
}

// ---- assembly of the coarse levels -------------------------------------------
// One thread per coarse node: its faces' coefficients (scale x the sum of the
// finer faces' in ascending order, the same bits from both sides), diagonal
// and pin, in FP64 with FP32 copies.
__device__ __forceinline__ void mg_node(const MgLevelArgs &a, int i)
{
    const int s = i >> 5, lane = i & 31;
    const int base = a.sp[s], w = (a.sp[s + 1] - base) >> 5;
    double diag = 0.0;
    // Two slots and four members of each in flight: a slot alone is a chain of
    // four dependent loads (face, list, member, coefficient).  One at a time the
    // assembly of the 256x128x128 box took 921 us, so 879; a mixed solve of the
    // 1024x512 tank with its assembly 3258 and 3243 us.
    for (int k = 0; k < w; k += 2) {
        int f[2], lo[2], hi[2], cl[2];
        double g[2] = {0.0, 0.0};
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int slot = base + (k + u) * kSlice + lane;
            f[u] = k + u < w ? a.face[slot] - 1 : -1;
            cl[u] = k + u < w ? a.col[slot] : 0;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            lo[u] = f[u] >= 0 ? a.mem_ptr[f[u]] : 0;
            hi[u] = f[u] >= 0 ? a.mem_ptr[f[u] + 1] : 0;
        }
        const int len = max(hi[0] - lo[0], hi[1] - lo[1]);
        for (int m = 0; m < len; m += 4) {
            int id[2][4];
            double v[2][4];
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q) id[u][q] = lo[u] + m + q < hi[u] ? a.mem[lo[u] + m + q] : -1;
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q) v[u][q] = id[u][q] >= 0 ? a.fine_gamma[id[u][q]] : 0.0;
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (id[u][q] >= 0) g[u] += v[u][q];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (k + u >= w) break;
            const int slot = base + (k + u) * kSlice + lane;
            if (f[u] >= 0) {
                g[u] *= a.scale[f[u]];
                if (cl[u] > i) a.gamma[f[u]] = g[u];
            }
            a.val64[slot] = g[u];
            a.val32[slot] = (float)g[u];
            diag += g[u];
        }
    }
    // the pin: the sum over the children's
    double pin = 0.0;
    const int c0 = a.cp[s], cw = (a.cp[s + 1] - c0) >> 5;
    for (int k = 0; k < cw; ++k) {
        const int ch = a.child[c0 + k * kSlice + lane];
        if (ch < 0) continue;
        if (a.fine_pin) pin += a.fine_pin[ch];
        else {
            const DevParams *p = a.stank ? a.tprm + a.stank[ch >> 5] : a.prm;
            if (ch == p->ref) pin += p->pin64;
        }
    }
    diag += pin;
    const double d = diag > 0.0 ? 1.0 / diag : 0.0;
    a.pin64[i] = pin;
    a.diag64[i] = diag;
    a.pin32[i] = (float)pin;
    a.dinv64[i] = d;
    a.dinv32[i] = (float)d;
}

__global__ void __launch_bounds__(256) k_mg_level(MgLevelArgs a)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.n_slices * kSlice) mg_node(a, i);
}

// Consecutive small levels, one CTA: each needs the finer one's coefficients.
// A launch each took 5 to 6 us, most of it latency.  The line lies at 256
// nodes, a row a thread: above it one SM's FP64 pipe costs more than the
// launch saves (at 2048 nodes the assembly of the 256x128x128 box took 876 us,
// at 256 it takes 869; the 1024x512 tank, assembled and solved, 3129 and 3112).
__global__ void __launch_bounds__(256) k_mg_small(MgSmallArgs a)
{
    for (int l = 0; l < a.n; ++l) {
        for (int i = threadIdx.x; i < a.lv[l].n_slices * kSlice; i += blockDim.x) mg_node(a.lv[l], i);
        __syncthreads();
    }
}

cudaError_t launch_mg_small(const MgSmallArgs &a, cudaStream_t s)
{
    k_mg_small<<<1, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_mg_level(const MgLevelArgs &a, cudaStream_t s)
{
    k_mg_level<<<(a.n_slices * kSlice + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

// Instantiations by precision, faces per row chunk and threads per CTA
// (*max_threads).  FP32: 1024 threads a CTA hide the gathers' latency where an
// SM has many rows; with few, what counts is the latency of some twenty grid
// barriers and of the tail's passes, which 512 threads pass faster.  601x203
// cells (25 slices an SM): 2.57 ms with 1024, 2.15 with 512; 1024x512 (108): 123
// and 127 us a V-cycle; 256x128x128 (862): 11.8 and 13.8 ms.
const void *mg_kernel(bool mixed, int max_width, int slices_per_sm, int *max_threads)
{
    const bool w4 = max_width <= 4;
    const bool wide = mixed && slices_per_sm > 64;
    *max_threads = wide ? 1024 : 512;
    if (wide) return w4 ? (const void *)k_solve_mg<float, 4, 1024, 1> : (const void *)k_solve_mg<float, 6, 1024, 1>;
    if (mixed) return w4 ? (const void *)k_solve_mg<float, 4, 512, 1> : (const void *)k_solve_mg<float, 6, 512, 1>;
    return w4 ? (const void *)k_solve_mg<double, 4, 512, 1> : (const void *)k_solve_mg<double, 6, 512, 1>;
}

}  // namespace gfm
