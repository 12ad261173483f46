// gfm_solve_csr_noalloc: FP64 Jacobi-PCG of a caller-held CSR system that
// allocates no device memory.
//
// Who needs it: code that runs inside a host program owning the device
// memory -- a CFD code or plugin whose memory comes from the host's pool or
// sits under a hard memory cap, where a cudaMalloc would be refused or would
// fragment the pool -- and time-critical loops in which cudaMalloc/cudaFree
// are off limits because they can synchronise the whole device.  Such a
// caller passes its own device arrays; every temporary the solve needs (the
// gathered CG vector, the per-CTA partial sums, the grid-barrier counter) lives in
// the file-scope array below, which the CUDA runtime places when it loads
// this library's device code on a GPU and keeps there until the process
// exits.
//
// The kernel is a persistent textbook Jacobi-preconditioned CG in FP64, a few
// rows per thread for the whole solve, restarted from the true residual when
// the recursive one claims convergence; the solve ends on the true residual
// only.  Two grid barriers per iteration, each closing a dot product: rows
// exchange (z, p_old) pairs and form their neighbours' p = z + beta p_old
// themselves, so the new direction needs no barrier of its own.  All vectors
// but the exchanged pairs, and the first entries of each row, stay in registers.
// What bounds it: the latency of the two barriers with their sums (about 3.5 us
// each) and the FP64 pipe, where a warp's instruction takes 64 cycles of a
// quarter SM: the sums are reduced in packed form (six adds for up to four
// values), the step lengths formed by one thread.  With three barriers, an
// error check at each and the vectors in memory an iteration took 19 us on
// 60 000 rows, 10.8 us now (31.1 -> 17.6 ms to a residual of 1e-12).  Forms
// with fewer sums were tried and dropped: pipelined CG (one barrier, 7.0 us) and
// Chronopoulos-Gear (7.9 us) lost accuracy on stretched cells, up to 25 000
// times the error at the same residual.
//
// All calls on a device share the one array, which keeps the last call's
// contents; the barrier block is cleared at every call, and every other word
// is written before it is read.  Two calls whose kernels overlap on the GPU
// (different streams, or different host threads) race on the array and corrupt
// each other's results: order them on one stream.
#include <cuda_runtime.h>

#include <cmath>
#include <mutex>

#include "gfm.h"

namespace {

constexpr int kMaxCells = GFM_NOALLOC_MAX_CELLS;
constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxGrid = 1024;
constexpr int kNR = 4;          // values per grid reduction
constexpr int kMaxChecks = 30;  // claims of convergence that the true residual may refute
constexpr int kMaxDevices = 256;

// Layout of the scratch array, in doubles.
constexpr size_t kCtl = 0;                                      // [32]: barrier counter (u64), error flag (int)
constexpr size_t kPart = 32;                                    // [2][kNR][kMaxGrid] per-CTA partial sums
constexpr size_t kVec = kPart + 2 * (size_t)kNR * kMaxGrid;     // the exchanged (z, p) pairs [kMaxCells]
constexpr size_t kScratchDoubles = kVec + 2 * (size_t)kMaxCells;  // 4.07 MiB at 262144 cells

static __device__ __align__(256) double g_noalloc_scratch[kScratchDoubles];

struct Args {
    int n, nnz;
    const int *rp, *col;
    const double *val, *b;
    double *x;
    double rtol;
    int max_iters, use_x0, G;
    unsigned long long budget_ns;
    gfm_solve_info *info;
    double *scr;
};

struct Bar {
    unsigned long long *count;
    int *err;
    double *part;
    unsigned long long budget, epoch;
    int G, parity;
};

struct Sh {
    double red[kWarps][kNR];
    double tot[kNR];
    double al, be;  // thread 0's step lengths
    int flag, act;
};

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void add_release(unsigned long long *p, unsigned long long v)
{
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Grid barrier on a monotone 64-bit arrival counter.  Every wait is bounded:
// past the budget the CTA records GFM_ERR_TIMEOUT and all CTAs return (one
// that waits sees the error flag).  With `check` an error that any CTA recorded
// before the barrier completed also stops every CTA; the flag is another round
// trip to L2, so the iterations go without.  False means the solve must stop.
__device__ bool bar_sync(Bar &g, Sh &sh, bool check = false)
{
    __syncthreads();
    g.epoch += 1;
    if (threadIdx.x == 0) {
        int fail = 0;
        add_release(g.count, 1ull);
        const unsigned long long target = g.epoch * (unsigned long long)g.G;
        unsigned long long t0 = 0;
        for (unsigned k = 0; load_acquire(g.count) < target; ++k) {
            const unsigned long long now = now_ns();
            if (k == 0) t0 = now;
            else if (now - t0 > g.budget) {
                atomicCAS(g.err, 0, (int)GFM_ERR_TIMEOUT);
                fail = 1;
                break;
            }
            if ((k & 15u) == 15u && *(volatile int *)g.err != 0) {
                fail = 1;
                break;
            }
        }
        if (check && *(volatile int *)g.err != 0) fail = 1;
        sh.flag = fail;
    }
    __syncthreads();
    return sh.flag == 0;
}

// The CTA's sums of NR <= 4 per-thread values, in a fixed order, to its
// partials.  Packed: the first two butterfly steps also halve the number of
// values a lane carries, so a warp spends six FP64 adds on four values.
template <int NR>
__device__ __forceinline__ void put_partials(const Bar &g, Sh &sh, const double (&v)[NR])
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto at = [&](int k) { return k < NR ? v[k < NR ? k : 0] : 0.0; };
    const bool h16 = (lane & 16) != 0, h8 = (lane & 8) != 0;
    double c = (h16 ? at(1) : at(0)) + __shfl_xor_sync(0xffffffffu, h16 ? at(0) : at(1), 16);
    if (NR > 2) {
        const double d = (h16 ? at(3) : at(2)) + __shfl_xor_sync(0xffffffffu, h16 ? at(2) : at(3), 16);
        c = (h8 ? d : c) + __shfl_xor_sync(0xffffffffu, h8 ? c : d, 8);
    } else {
        c += __shfl_xor_sync(0xffffffffu, c, 8);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    if ((lane & 7) == 0) {  // lanes 0, 16, 8, 24 hold values 0, 1, 2, 3
        const int k = (h8 ? 2 : 0) + (h16 ? 1 : 0);
        if (k < NR) sh.red[warp][k] = c;
    }
    __syncthreads();
    if (warp < NR) {
        double t = lane < kWarps ? sh.red[lane][warp] : 0.0;
#pragma unroll
        for (int o = kWarps / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) g.part[((size_t)g.parity * kNR + warp) * kMaxGrid + blockIdx.x] = t;
    }
}

// After the barrier: warp k < NR adds value k over all CTAs, bitwise alike in
// every CTA, into sh.tot[k].  The caller synchronises the CTA.
template <int NR>
__device__ __forceinline__ void take_sums(Bar &g, Sh &sh)
{
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (warp < NR) {
        const double *src = g.part + ((size_t)g.parity * kNR + warp) * kMaxGrid;
        double v[8], t = 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = lane + 32 * q < g.G ? __ldcg(src + lane + 32 * q) : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (32 * q < g.G) t += v[q];
        for (int c = lane + 256; c < g.G; c += 32) t += __ldcg(src + c);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) sh.tot[warp] = t;
    }
    g.parity ^= 1;
}

template <int NR>
__device__ bool grid_sum(Bar &g, Sh &sh, const double (&v)[NR])
{
    put_partials<NR>(g, sh, v);
    if (!bar_sync(g, sh)) return false;
    take_sums<NR>(g, sh);
    __syncthreads();
    return true;
}

__device__ void write_info(const Args &a, int iters, int checks, int status, double l2, double l1)
{
    if (a.info == nullptr || blockIdx.x != 0 || threadIdx.x != 0) return;
    a.info->iters = iters;
    a.info->refinements = checks;
    a.info->status = status;
    a.info->reserved = 0;
    a.info->rel_res_l2 = l2;
    a.info->rel_res_l1 = l1;
}

// The rows of a thread: row r is base + r * kThreads; the first W entries of
// each in registers.
template <int R, int W>
struct Rows {
    static constexpr int UR = R <= 4 ? R : 1;  // many rows: loops over local arrays
    int i0, n;
    int e0[R], e1[R];
    double cv[R][W > 0 ? W : 1];
    int cc[R][W > 0 ? W : 1];
    __device__ __forceinline__ int row(int r) const { return i0 + r * kThreads; }
    __device__ __forceinline__ bool on(int r) const { return row(r) < n; }
    // (A v)_row for every row of the thread, v_j = get(j) read from memory that
    // other CTAs write: the gathers of all rows' cached entries in flight together
    template <typename Get>
    __device__ __forceinline__ void product(const Args &a, Get get, double (&out)[R]) const
    {
        double g[R][W > 0 ? W : 1];
#pragma unroll UR
        for (int r = 0; r < R; ++r)
#pragma unroll
            for (int k = 0; k < W; ++k) g[r][k] = e0[r] + k < e1[r] ? get(cc[r][k]) : 0.0;
#pragma unroll UR
        for (int r = 0; r < R; ++r) {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < W; ++k) s = fma(cv[r][k], g[r][k], s);
            for (int e = e0[r] + W; e < e1[r]; ++e) s = fma(__ldg(a.val + e), get(__ldg(a.col + e)), s);
            out[r] = s;
        }
    }
};

enum : int { kGo = 0, kVerify = 1, kStop = 2 };

template <int R, int W>
__global__ void __launch_bounds__(kThreads, 1) k_pcg_csr_noalloc(Args a)
{
    constexpr int UR = R <= 4 ? R : 1;
    __shared__ Sh sh;
    Bar g{reinterpret_cast<unsigned long long *>(a.scr + kCtl), reinterpret_cast<int *>(a.scr + kCtl + 1),
          a.scr + kPart, a.budget_ns, 0ull, a.G, 0};
    double2 *zp = reinterpret_cast<double2 *>(a.scr + kVec);
    const int n = a.n;
    const double rtol2 = a.rtol * a.rtol;
    int iters = 0, checks = 0, status = GFM_ERR_NOT_CONVERGED;
    Rows<R, W> rows;
    rows.i0 = blockIdx.x * kThreads * R + threadIdx.x;
    rows.n = n;
    double x[R], r[R], z[R], p[R], d[R], t[R];

    // Validate the caller's CSR structure before any vector is gathered
    // through it: 0 <= row_ptr[i] <= row_ptr[i+1] <= nnz and 0 <= col < n.
    // A row with bad bounds is skipped, so the check itself reads only
    // row_ptr [n+1] and, within checked bounds, col/val [nnz].  Jacobi
    // weights from the diagonal entries; a row without a positive one is an
    // argument error too.  Start vector.  Every row is checked by some CTA
    // before the barrier, and any error stops every CTA after it.
    int bad = 0;
#pragma unroll UR
    for (int k = 0; k < R; ++k) {
        const int i = rows.row(k);
        rows.e0[k] = rows.e1[k] = 0;
        x[k] = d[k] = 0.0;
#pragma unroll
        for (int m = 0; m < W; ++m) {
            rows.cv[k][m] = 0.0;
            rows.cc[k][m] = 0;
        }
        if (!rows.on(k)) continue;
        const int e0 = a.rp[i], e1 = a.rp[i + 1];
        double dg = 0.0;
        if (e0 < 0 || e1 < e0 || e1 > a.nnz) {
            bad = 1;
        } else {
            for (int e = e0; e < e1; ++e) {
                const int c = a.col[e];
                if (c < 0 || c >= n) bad = 1;
                else if (c == i) dg += a.val[e];
            }
            rows.e0[k] = e0;
            rows.e1[k] = e1;
#pragma unroll
            for (int m = 0; m < W; ++m)
                if (e0 + m < e1) {
                    rows.cv[k][m] = a.val[e0 + m];
                    rows.cc[k][m] = a.col[e0 + m];
                }
        }
        if (!(dg > 0.0) || !isfinite(dg)) bad = 1;
        d[k] = 1.0 / dg;
        if (a.use_x0) x[k] = a.x[i];
        else a.x[i] = 0.0;
    }
    if (bad) atomicCAS(g.err, 0, (int)GFM_ERR_ARG);
    if (!bar_sync(g, sh, true)) {
        write_info(a, iters, checks, *(volatile int *)g.err, -1.0, -1.0);
        return;
    }
    // t = b - A x (x settled in the caller's array)
    auto residual = [&]() {
        rows.product(a, [&](int c) { return __ldcg(a.x + c); }, t);
#pragma unroll UR
        for (int k = 0; k < R; ++k) t[k] = rows.on(k) ? a.b[rows.row(k)] - t[k] : 0.0;
    };

    double bb = 0.0;
    bool aborted = false;
    // one round: the true residual, then iterations until it claims convergence
    for (;;) {
        if (checks > 0) {
#pragma unroll UR
            for (int k = 0; k < R; ++k)
                if (rows.on(k)) a.x[rows.row(k)] = x[k];
            if (!bar_sync(g, sh)) { aborted = true; break; }
        }
        residual();
        double v[3] = {0.0, 0.0, 0.0};
#pragma unroll UR
        for (int k = 0; k < R; ++k) {
            r[k] = t[k];
            z[k] = d[k] * r[k];
            p[k] = 0.0;
            v[0] = fma(r[k], r[k], v[0]);
            v[1] = fma(r[k], z[k], v[1]);
            if (rows.on(k)) {
                const double bi = a.b[rows.row(k)];
                v[2] = fma(bi, bi, v[2]);
                zp[rows.row(k)] = make_double2(z[k], 0.0);
            }
        }
        if (!grid_sum<3>(g, sh, v)) { aborted = true; break; }
        const double rr = sh.tot[0];
        double rz = sh.tot[1];  // thread 0's
        bb = sh.tot[2];
        ++checks;
        if (bb == 0.0) {  // b = 0: the solution is 0
#pragma unroll UR
            for (int k = 0; k < R; ++k) x[k] = 0.0;
            status = GFM_OK;
            break;
        }
        if (!isfinite(rr)) { status = GFM_ERR_BREAKDOWN; break; }
        if (rr <= rtol2 * bb) { status = GFM_OK; break; }
        if (iters >= a.max_iters || checks > kMaxChecks) break;
        double be = 0.0;
        bool stop = false;
        for (;;) {
            // p = z + beta p here and, from their pairs, in the neighbours; q = A p, p.q
            rows.product(a, [&](int c) {
                const double2 v = __ldcg(zp + c);
                return fma(be, v.y, v.x);
            }, t);
            double c[1] = {0.0};
#pragma unroll UR
            for (int k = 0; k < R; ++k) {
                p[k] = fma(be, p[k], z[k]);
                c[0] = fma(p[k], t[k], c[0]);
            }
            if (!grid_sum<1>(g, sh, c)) { aborted = true; break; }
            if (threadIdx.x == 0) {
                const double pq = sh.tot[0];
                const bool ok = pq > 0.0 && isfinite(pq);
                sh.act = ok ? kGo : kStop;
                sh.al = ok ? rz / pq : 0.0;
            }
            __syncthreads();
            if (sh.act == kStop) { status = GFM_ERR_BREAKDOWN; stop = true; break; }
            const double al = sh.al;
            double u[2] = {0.0, 0.0};
#pragma unroll UR
            for (int k = 0; k < R; ++k) {
                x[k] = fma(al, p[k], x[k]);
                r[k] = fma(-al, t[k], r[k]);
                z[k] = d[k] * r[k];
                if (rows.on(k)) zp[rows.row(k)] = make_double2(z[k], p[k]);
                u[0] = fma(r[k], r[k], u[0]);
                u[1] = fma(r[k], z[k], u[1]);
            }
            if (!grid_sum<2>(g, sh, u)) { aborted = true; break; }
            ++iters;
            if (threadIdx.x == 0) {
                sh.act = sh.tot[0] <= rtol2 * bb || iters >= a.max_iters ? kVerify : kGo;
                sh.be = sh.tot[1] / rz;
                rz = sh.tot[1];
            }
            __syncthreads();
            if (sh.act != kGo) break;
            be = sh.be;
        }
        if (aborted || stop) break;
    }
    if (aborted) {
        write_info(a, iters, checks, *(volatile int *)g.err, -1.0, -1.0);
        return;
    }

    // final record: true residual (L2, and the normalised L1 residual with
    // the row sums of A applied to the mean of x)
    {
#pragma unroll UR
        for (int k = 0; k < R; ++k)
            if (rows.on(k)) a.x[rows.row(k)] = x[k];
        bool ok = bar_sync(g, sh);
        double v[3] = {0.0, 0.0, 0.0};
        if (ok) {
            residual();
#pragma unroll UR
            for (int k = 0; k < R; ++k)
                if (rows.on(k)) {
                    const double bi = a.b[rows.row(k)];
                    v[0] = fma(t[k], t[k], v[0]);
                    v[1] += x[k];
                    v[2] = fma(bi, bi, v[2]);
                }
            ok = grid_sum<3>(g, sh, v);
        }
        double rr = 0.0, xavg = 0.0, bs = 0.0, l1[2] = {0.0, 0.0};
        if (ok) {
            rr = sh.tot[0];
            xavg = sh.tot[1] / (double)n;
            bs = sh.tot[2];
#pragma unroll UR
            for (int k = 0; k < R; ++k)
                if (rows.on(k)) {
                    double rs = 0.0;
                    for (int e = rows.e0[k]; e < rows.e1[k]; ++e) rs += a.val[e];
                    const double bi = a.b[rows.row(k)], ax = bi - t[k];
                    l1[0] += fabs(t[k]);
                    l1[1] += fabs(ax - xavg * rs) + fabs(bi - xavg * rs);
                }
            __syncthreads();  // the totals above are read before they are replaced
            ok = grid_sum<2>(g, sh, l1);
        }
        if (ok) write_info(a, iters, checks, status, bs > 0.0 ? sqrt(rr / bs) : 0.0, sh.tot[0] / (sh.tot[1] + 1e-300));
        else write_info(a, iters, checks, *(volatile int *)g.err, -1.0, -1.0);
    }
}

// Rows per thread: the fewest that hold n rows on the device's co-resident
// grid (each row's vectors live in registers); the largest, whose arrays go to
// local memory, only serves devices with few SMs.
const void *pick_kernel(int n, int sms, int *rows)
{
    const long long per = (long long)sms * kThreads;
    if (n <= per) { *rows = 1; return (const void *)k_pcg_csr_noalloc<1, 7>; }
    if (n <= 2 * per) { *rows = 2; return (const void *)k_pcg_csr_noalloc<2, 5>; }
    if (n <= 4 * per) { *rows = 4; return (const void *)k_pcg_csr_noalloc<4, 0>; }
    *rows = 16;
    return (const void *)k_pcg_csr_noalloc<16, 0>;
}

struct DeviceScratch {
    double *ptr = nullptr;
    int sms = 0;
};

std::mutex g_mu;
DeviceScratch g_dev[kMaxDevices];

// One-time set-up on the current device: the device address of the scratch
// array (this also loads the device code if the runtime loads it lazily) and
// the SM count (one co-resident CTA each).
gfm_status setup_current_device(DeviceScratch &out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return GFM_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return GFM_ERR_ARG;
    std::lock_guard<std::mutex> lock(g_mu);
    DeviceScratch &d = g_dev[dev];
    if (d.ptr == nullptr) {
        void *ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || ptr == nullptr) return GFM_ERR_CUDA;
        int coop = 0, sms = 0;
        if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop)
            return GFM_ERR_CUDA;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            return GFM_ERR_CUDA;
        // load every instantiation now: a first call may not load code under capture
        for (int rows = 1; rows <= 16; rows *= 2) {
            int r = 0, per_sm = 0;
            const void *k = pick_kernel(rows * sms * kThreads, sms, &r);
            if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, 0) != cudaSuccess || per_sm < 1)
                return GFM_ERR_CUDA;
        }
        d.sms = sms < kMaxGrid ? sms : kMaxGrid;
        d.ptr = static_cast<double *>(ptr);
    }
    out = d;
    return GFM_OK;
}

}  // namespace

extern "C" gfm_status gfm_solve_csr_noalloc(int32_t n, int32_t nnz, const int32_t *row_ptr, const int32_t *col,
                                            const double *val, const double *b, double *x, double rtol,
                                            int32_t max_iters, int32_t use_x0, double timeout_ms,
                                            gfm_solve_info *info, gfm_stream stream)
{
    if (n < 1 || n > kMaxCells) return GFM_ERR_ARG;  // beyond the fixed scratch capacity
    if (nnz < n) return GFM_ERR_ARG;                  // every row needs its diagonal entry
    if (!row_ptr || !col || !val || !b || !x) return GFM_ERR_ARG;
    if (!(rtol > 0.0) || !std::isfinite(rtol) || max_iters < 0 || !(timeout_ms > 0.0) || !std::isfinite(timeout_ms))
        return GFM_ERR_ARG;
    (void)cudaGetLastError();  // a non-sticky error left by earlier, unrelated work
    DeviceScratch d;
    const gfm_status st = setup_current_device(d);
    if (st != GFM_OK) return st;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    int rows = 1;
    const void *kernel = pick_kernel(n, d.sms, &rows);
    const int want = (n + kThreads * rows - 1) / (kThreads * rows);
    if (want > d.sms) return GFM_ERR_CUDA;
    Args a;
    a.n = n;
    a.nnz = nnz;
    a.rp = row_ptr;
    a.col = col;
    a.val = val;
    a.b = b;
    a.x = x;
    a.rtol = rtol;
    a.max_iters = max_iters;
    a.use_x0 = use_x0 ? 1 : 0;
    a.G = want;
    const double ns = timeout_ms * 1e6;
    a.budget_ns = ns > 1.8e19 ? 18000000000000000000ull : (unsigned long long)ns;
    a.info = info;
    a.scr = d.ptr;
    if (cudaMemsetAsync(d.ptr + kCtl, 0, 32 * sizeof(double), s) != cudaSuccess) return GFM_ERR_CUDA;
    void *args[] = {&a};
    if (cudaLaunchCooperativeKernel(kernel, dim3(a.G), dim3(kThreads), args, 0, s) !=
        cudaSuccess)
        return GFM_ERR_CUDA;
    return GFM_OK;
}
