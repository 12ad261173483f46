// isoAdvector advection step (Sec. 3.2): the heavy-fluid volume each face
// passes during a time step, and the volume-fraction update.
//
// Over [t, t + dt] the face passes dV_f = phi_f int alpha_f+(tau) dtau
// (Eq. dV), alpha_f+ being the submerged fraction of the face (Eq. alphaf).
// In the upwind cell the interface is the isoface plane (centre x_S, unit
// normal n_S away from the heavy fluid) moving at normal speed U_S.n_S, so a
// point x is reached at t_x = (x - x_S).n_S / U_S.n_S (Eq. tv).  The face is
// the union of triangles (face centre, v_k, v_k+1).  On each triangle with
// vertex times t1 <= t2 <= t3 the sweep line enters at x1, passes x2 while
// cutting edge 1-3 at x4 (Eq. x_41), and leaves at x3; the swept fraction is
// quadratic in tau on [t1, t2] and on [t2, t3] (Eqs. aplus1, aplus2) with
//     a2 = |x41 x x21| / 2A = (t2 - t1)/(t3 - t1)   (the swept fraction at t2),
//     F  = a2 ((tau - t1)/(t2 - t1))^2              on [t1, t2],
//     F  = 1 - (1 - a2) ((t3 - tau)/(t3 - t2))^2    on [t2, t3],
// and the time integral over [0, dt] is the sum of the pieces' exact
// integrals (Eq. intaplus), written in shifted form for conditioning.  When
// the interface moves towards the heavy fluid (U_S.n_S < 0) the swept part
// is the part that has drained: the submerged fraction is 1 - F.  A face
// whose upwind cell has no isoface carries that cell's alpha throughout.
//
// A thread per face and a lane per triangle (FP64 geometry); then one thread
// per cell sums its faces' volumes in ascending face order:
//     alpha_P(t + dt) = alpha_P(t) - 1/V_P sum_f s_Pf dV_f.
#include "gfm_internal.h"

namespace gfm {

namespace {

struct V3 {
    double x, y, z;
};

__device__ __forceinline__ V3 sub3(V3 a, V3 b) { return V3{a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ double cross_norm(V3 a, V3 b)
{
    const double cx = a.y * b.z - a.z * b.y, cy = a.z * b.x - a.x * b.z, cz = a.x * b.y - a.y * b.x;
    return sqrt(cx * cx + cy * cy + cz * cz);
}

// The sweep of one triangle: ordered vertex times.  x4 lies on edge 1-3 where
// the sweep is at t2 (Eq. x_41: x41 = r x31, r = (t2 - t1)/(t3 - t1)), so the
// swept fraction at t2 is |r x31 x x21| / |x31 x x21| = r.
struct Sweep {
    double t1, t2, t3;
};

__device__ __forceinline__ Sweep make_sweep(double a, double b, double c)
{
    const double lo = fmin(a, b), hi = fmax(a, b);
    return Sweep{fmin(lo, c), fmax(lo, fmin(hi, c)), fmax(hi, c)};
}

// The swept fraction F(tau) (Eqs. aplus1, aplus2).
__device__ double sweep_at(const Sweep &w, double tau)
{
    if (tau <= w.t1) return 0.0;
    if (tau >= w.t3) return 1.0;
    const double t31 = w.t3 - w.t1;
    if (tau <= w.t2) {
        const double u = tau - w.t1;
        return (u / (w.t2 - w.t1)) * (u / t31);
    }
    const double u = w.t3 - tau;
    return 1.0 - (u / (w.t3 - w.t2)) * (u / t31);
}

// int_0^dt F(tau) dtau: the exact integrals of the quadratic pieces clipped
// to [0, dt] (Eq. intaplus, in shifted form).  With a2 = (t2 - t1)/(t3 - t1)
// the pieces' factors a2/(3 (t2 - t1)^2) and (1 - a2)/(3 (t3 - t2)^2) are
// 1/(3 (t2 - t1)(t3 - t1)) and 1/(3 (t3 - t2)(t3 - t1)).
__device__ double sweep_integral(const Sweep &w, double dt)
{
    double I = 0.0;
    const double t31 = 3.0 * (w.t3 - w.t1);
    {  // [t1, t2]: a2 ((tau - t1)/(t2 - t1))^2
        const double lo = fmin(fmax(0.0, w.t1), w.t2), hi = fmin(fmax(dt, w.t1), w.t2);
        if (hi > lo) {
            const double d = w.t2 - w.t1, u = hi - w.t1, l = lo - w.t1;
            I += (u * u * u - l * l * l) / (d * t31);
        }
    }
    {  // [t2, t3]: 1 - (1 - a2) ((t3 - tau)/(t3 - t2))^2
        const double lo = fmin(fmax(0.0, w.t2), w.t3), hi = fmin(fmax(dt, w.t2), w.t3);
        if (hi > lo) {
            const double d = w.t3 - w.t2, u = w.t3 - lo, l = w.t3 - hi;
            I += (hi - lo) - (u * u * u - l * l * l) / (d * t31);
        }
    }
    const double s3 = fmax(0.0, w.t3);  // [t3, dt]: fully swept
    if (dt > s3) I += dt - s3;
    return I;
}

// A block takes 256 faces.  First every thread settles its face if the upwind
// cell has no isoface (most faces of a flow); the others' numbers are packed
// into a list, on which groups of four lanes work, a triangle per lane.  What
// bounds the second part is the FP64 pipe (a warp's FP64 instruction takes as
// long with one lane active as with 32): with one thread per face, nearly
// every warp ran all four triangles of a quad for its one face in ten that
// needs them.  2.27M faces, one in ten with an isoface: 2480 -> 333 us.
__global__ void __launch_bounds__(256) k_iso_flux(IsoArgs a)
{
    __shared__ int list[256];
    __shared__ int wcount[8];
    const int f0 = blockIdx.x * 256;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t n = (size_t)a.n, F = (size_t)a.F, nvt = (size_t)a.nvt;
    bool iso = false;
    {
        const int f = f0 + threadIdx.x;
        if (f < a.F) {
            const double ph = a.phi[f];
            const int U = ph >= 0.0 ? a.owner[f] : a.neighbour[f];
            iso = a.has_iso[U] != 0;
            if (!iso) {
                const double I = a.alpha[U] * a.dt;
                if (a.integral) a.integral[f] = I;
                a.dV[f] = ph * I;
            }
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, iso);
    if (lane == 0) wcount[warp] = __popc(m);
    __syncthreads();
    int before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        before += w < warp ? wcount[w] : 0;
        total += wcount[w];
    }
    if (iso) list[before + __popc(m & ((1u << lane) - 1u))] = f0 + threadIdx.x;
    __syncthreads();
    const int sub = threadIdx.x & 3;
    const unsigned group = 0xFu << (lane & 28);
    for (int q = threadIdx.x >> 2; q < total; q += 64) {
        const int f = list[q];
        const double ph = a.phi[f];
        const int U = ph >= 0.0 ? a.owner[f] : a.neighbour[f];
        const V3 xs{a.xS[U], a.xS[n + U], a.xS[2 * n + U]};
        const V3 ns{a.nS[U], a.nS[n + U], a.nS[2 * n + U]};
        const double un = a.UnS[U];
        const V3 c{a.xf[f], a.xf[F + f], a.xf[2 * F + f]};
        const int v0 = a.fv_ptr[f], nv = a.fv_ptr[f + 1] - v0;
        // a static interface (U_S.n_S = 0): the fraction behind the plane,
        // the sweep read at tau = 0 with the signed distances as times
        const bool moving = un != 0.0;
        const double iu = moving ? 1.0 / un : 1.0;
        const double tc = dot(sub3(c, xs), ns) * iu;
        double atot = 0.0, acc = 0.0;
        for (int e0 = 0; e0 < nv; e0 += 4) {
            const int e = e0 + sub;
            if (e < nv) {
                const int i0 = v0 + e, i1 = v0 + (e + 1 < nv ? e + 1 : 0);
                const V3 pa{a.fv_xyz[i0], a.fv_xyz[nvt + i0], a.fv_xyz[2 * nvt + i0]};
                const V3 pb{a.fv_xyz[i1], a.fv_xyz[nvt + i1], a.fv_xyz[2 * nvt + i1]};
                const double at = cross_norm(sub3(pa, c), sub3(pb, c));  // twice the area
                if (at > 0.0) {
                    const Sweep w = make_sweep(tc, dot(sub3(pa, xs), ns) * iu, dot(sub3(pb, xs), ns) * iu);
                    double sw;
                    if (!moving) sw = sweep_at(w, 0.0) * a.dt;
                    else {
                        sw = sweep_integral(w, a.dt);
                        if (un < 0.0) sw = a.dt - sw;  // moving into the heavy fluid: the swept part has drained
                    }
                    atot += at;
                    acc += at * sw;
                }
            }
        }
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
            atot += __shfl_xor_sync(group, atot, off);
            acc += __shfl_xor_sync(group, acc, off);
        }
        if (sub == 0) {
            const double I = atot > 0.0 ? acc / atot : 0.0;
            if (a.integral) a.integral[f] = I;
            a.dV[f] = ph * I;
        }
    }
}

__global__ void __launch_bounds__(256) k_iso_cells(IsoArgs a)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.n) return;
    const int base = a.cf.ptr[c >> 5], w = (a.cf.ptr[(c >> 5) + 1] - base) >> 5, lane = c & 31;
    double acc = 0.0;
    for (int k0 = 0; k0 < w; k0 += 3) {
        int code[3];
        double v[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) code[q] = k0 + q < w ? a.cf.face[base + (k0 + q) * kSlice + lane] : 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) v[q] = code[q] != 0 ? a.dV[(code[q] > 0 ? code[q] : -code[q]) - 1] : 0.0;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (code[q] != 0) acc = code[q] > 0 ? acc + v[q] : acc - v[q];
    }
    a.alpha_new[c] = a.alpha[c] - acc / a.V[c];
}

}  // namespace

cudaError_t launch_iso(const IsoArgs &a, cudaStream_t s)
{
    if (a.F > 0) k_iso_flux<<<(a.F + 255) / 256, 256, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || !a.alpha_new) return e;
    k_iso_cells<<<(a.n + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace gfm
