// Dynamic-pressure gradient of the momentum equation and cell velocities
// from face fluxes (Sec. 3.1, Eq. 20 and the paragraph after it; Eq. 2's
// pressure term, Eq. 8).
//
// The momentum equation needs (1/rho) grad p_d at cell centres.  By the
// Gauss theorem with linear cell-to-face interpolation, cell P sees face f
// through p_f = w_P p_P + (1 - w_P) pN~, where pN~ is the neighbour's value,
// replaced at an interface face by its ghost value extrapolated into P's
// fluid (Eq. 20 from the wet side, the analogous expression from the dry
// side).  Written out, both ghost values collapse onto the coefficients the
// assembly already holds:
//     beta_P (pN~ - p_P) = (p_N - p_P - s_Pf J_f) / rho_f,
//     rho_f = lambda_f rho_w + (1 - lambda_f) rho_a   (the harmonic face density of Eq. 18),
// J_f the oriented jump (Eq. 7) and s_Pf = +1 if P owns f, -1 otherwise; off
// the interface J_f = 0 and rho_f is the phase's own density.  With
// zero-gradient walls the face sum reduces to the internal faces in
// difference form, so
//     (1/rho grad p_d)_P = 1/V_P sum_f (1 - w_P) (p_N - p_P - s_Pf J_f) / rho_f  s_Pf S_f,
//     (1 - w_P) = S_f.(x_f - x_P) / S_f.(x_N - x_P).
// The reconstruction of a cell velocity from face fluxes uses the identity
// sum_f (u.S_f)(x_f - x_P) = V_P u of a closed cell:
//     U_P = 1/V_P sum_f s_Pf phi_f (x_f - x_P).
//
// Two passes, FP64 throughout, both in the caller's order.  k_grad_faces, a
// thread per face, reads every face array once and coalesced and leaves what
// both cells need in one 32-byte record per face and quantity:
//     q_f S_f and (1 - w_own),  q_f = (p_N - p_O - J_f) / rho_f,
// (both sides of a face see the same q_f S_f: s_Pf and the sign of the
// difference cancel; 1 - w_nb = w_own), and the face centre and flux.  S.d and
// its inverse are the mesh's and come from a table, so the neighbour's p_d is
// the one random gather.  k_grad_cells, a thread per cell, sums its faces'
// records in ascending face order; the caller's order keeps its outputs and,
// where faces are sorted by owner, half of its records coalesced.  With one
// pass over the cells in internal order every face was evaluated twice, on an
// FP64 pipe that bounds the work on meshes that stay in L2, and each of its
// dozen face and neighbour values was a gather of its own: in a random cell
// order each costs a whole DRAM granule.  201x101x99 cells in a random order,
// gradient and velocity: 2090 -> 757 us (1410 with the cells in internal
// order and both centres gathered by the face pass).
#include "gfm_div.cuh"
#include "gfm_internal.h"

namespace gfm {

namespace {

// A whole record in one 32-byte access (sm_100 and later), a full sector.
__device__ __forceinline__ void store_record(double4 *p, double x, double y, double z, double w)
{
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(x), "d"(y), "d"(z), "d"(w) : "memory");
}
__device__ __forceinline__ double4 load_record(const double4 *p)
{
    double4 v;
    asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v.x), "=d"(v.y), "=d"(v.z), "=d"(v.w) : "l"(p));
    return v;
}

// S.(x_f - x_own) / S.d of a face with a given centre.
__device__ __forceinline__ double face_weight(const GradArgs &a, int f, int o, double S0, double S1, double S2,
                                              double x0, double x1, double x2)
{
    const size_t n = (size_t)a.n;
    const double2 sd = a.sd[f];
    return div_known(S0 * (x0 - a.C[o]) + S1 * (x1 - a.C[n + o]) + S2 * (x2 - a.C[2 * n + o]), sd.x, sd.y);
}

// The densities of a face's tank and their inverses as div_known takes them.
struct Densities {
    double w, a, inv_w, inv_a;
};
__device__ __forceinline__ Densities densities(const GradArgs &a, int f)
{
    if (!a.ftank) return Densities{a.rho_w, a.rho_a, a.inv_w, a.inv_a};
    const TankPhys *tp = a.tphys + a.ftank[f];
    return Densities{tp->rho_w, tp->rho_a, tp->inv_w, tp->inv_a};
}

template <bool G, bool U>
__global__ void __launch_bounds__(256) k_grad_faces(GradArgs a)
{
    // faces on the interface, packed: their general division is the dearest
    // part, and in a random cell order nearly every warp holds one of them
    __shared__ int list[256];
    __shared__ double val[256];
    __shared__ int wcount[8];
    const int f = blockIdx.x * 256 + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t n = (size_t)a.n, F = (size_t)a.F;
    const bool on = f < a.F;
    const int o = on ? a.owner[f] : 0, nb = on ? a.neighbour[f] : 0;
    double q = 0.0;
    if (G) {
        bool iface = false;
        if (on) {
            const int8_t kind = a.kind[f];
            iface = kind > 1;  // 0: both cells dry, 1: both wet
            q = a.p[nb] - a.p[o];
            if (iface) {
                q -= a.jump[f];
            } else {
                const Densities rho = densities(a, f);
                q = div_known(q, kind ? rho.w : rho.a, kind ? rho.inv_w : rho.inv_a);
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, iface);
        if (lane == 0) wcount[warp] = __popc(m);
        __syncthreads();
        int before = 0, total = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            before += w < warp ? wcount[w] : 0;
            total += wcount[w];
        }
        if (total > 0) {
            const int at = before + __popc(m & ((1u << lane) - 1u));
            if (iface) {
                list[at] = f;
                val[at] = q;
            }
            __syncthreads();
            if ((int)threadIdx.x < total) {
                const int e = list[threadIdx.x];
                const double lam = a.lambda[e];
                const Densities rho = densities(a, e);
                val[threadIdx.x] = val[threadIdx.x] / (lam * rho.w + (1.0 - lam) * rho.a);
            }
            __syncthreads();
            if (iface) q = val[at];
        }
    }
    if (!on) return;
    double4 *rec = a.rec + (size_t)f * ((int)G + (int)U);
    const bool mid = !a.xf;
    double x0 = 0.0, x1 = 0.0, x2 = 0.0;
    if (!mid) {
        x0 = a.xf[f];
        x1 = a.xf[F + f];
        x2 = a.xf[2 * F + f];
    }
    if (G) {
        const double S0 = a.Sf[f], S1 = a.Sf[F + f], S2 = a.Sf[2 * F + f];
        const double fac = mid ? 0.5 : face_weight(a, f, o, S0, S1, S2, x0, x1, x2);
        store_record(rec, q * S0, q * S1, q * S2, fac);
    }
    if (U) {
        const double ph = a.phi[f];
        if (mid) {
            // without face centres x_f - x_P is half the centre distance, the
            // same for both cells but for the sign, which the flux's cancels
            const double h = 0.5 * ph;
            store_record(rec + (int)G, h * (a.C[nb] - a.C[o]), h * (a.C[n + nb] - a.C[n + o]),
                         h * (a.C[2 * n + nb] - a.C[2 * n + o]), ph);
        } else {
            store_record(rec + (int)G, x0, x1, x2, ph);
        }
    }
}

// Both passes in one launch, for small meshes: a block takes a slice of 32
// cells, eight lanes a cell.  Each lane evaluates one face as k_grad_faces does
// (a face is evaluated for both its cells, but all faces of a cell at once), and
// six threads a cell, one a component, sum the faces in ascending order as
// k_grad_cells does: the same bits.  Such a call is bound by the host's launches
// and the passes' latency.  Gradient and velocity, us on the device, two
// launches and one: 10.0 and 5.2 (800 cells), 13.8 and 10.7 (24x18x12), 11.0 and
// 9.8 (200x60), 16.3 and 15.2 (30x24x20: 41,400 faces), 12.1 and 17.1 (300x90:
// 53,610 faces), where evaluating every face twice costs more; called from
// Python one after another 33 and 29.  The line lies at 45,056 faces.
template <bool G, bool U>
__global__ void __launch_bounds__(256) k_grad_small(GradArgs a)
{
    __shared__ double part[8][8][33];  // [slot][weight, q S; flux, x][cell]
    __shared__ int code[8][32];
    const size_t n = (size_t)a.n, F = (size_t)a.F;
    const int base = a.cf.ptr[blockIdx.x], w = (a.cf.ptr[blockIdx.x + 1] - base) >> 5;
    const int c = threadIdx.x >> 3, k = threadIdx.x & 7;
    const int comp = threadIdx.x >> 5, lane = threadIdx.x & 31, cell = blockIdx.x * 32 + lane;
    const bool sums = cell < a.n && ((G && comp < 3) || (U && comp >= 3 && comp < 6));
    double acc = 0.0, xP = 0.0, iv = 0.0;
    if (sums) {
        iv = 1.0 / a.V[cell];
        if (comp >= 3 && a.xf) xP = a.C[(size_t)(comp - 3) * n + cell];
    }
    for (int k0 = 0; k0 < w; k0 += 8) {
        const int fo = k0 + k < w && (int)blockIdx.x * 32 + c < a.n ? a.cf.face[base + (k0 + k) * kSlice + c] : 0;
        code[k][c] = fo;
        if (fo != 0) {
            const int f = (fo > 0 ? fo : -fo) - 1, o = a.owner[f], nb = a.neighbour[f];
            double x0 = 0.0, x1 = 0.0, x2 = 0.0;
            if (a.xf) {
                x0 = a.xf[f];
                x1 = a.xf[F + f];
                x2 = a.xf[2 * F + f];
            }
            if (G) {
                const int8_t kind = a.kind[f];
                const Densities rho = densities(a, f);
                double q = a.p[nb] - a.p[o];
                if (kind > 1) {
                    const double lam = a.lambda[f];
                    q -= a.jump[f];
                    q = q / (lam * rho.w + (1.0 - lam) * rho.a);
                } else {
                    q = div_known(q, kind ? rho.w : rho.a, kind ? rho.inv_w : rho.inv_a);
                }
                const double S0 = a.Sf[f], S1 = a.Sf[F + f], S2 = a.Sf[2 * F + f];
                const double fac = a.xf ? face_weight(a, f, o, S0, S1, S2, x0, x1, x2) : 0.5;
                part[k][0][c] = fo > 0 ? fac : 1.0 - fac;
                part[k][1][c] = q * S0;
                part[k][2][c] = q * S1;
                part[k][3][c] = q * S2;
            }
            if (U) {
                const double ph = a.phi[f];
                if (a.xf) {
                    part[k][4][c] = fo > 0 ? ph : -ph;
                    part[k][5][c] = x0;
                    part[k][6][c] = x1;
                    part[k][7][c] = x2;
                } else {
                    const double h = 0.5 * ph;
                    part[k][5][c] = h * (a.C[nb] - a.C[o]);
                    part[k][6][c] = h * (a.C[n + nb] - a.C[n + o]);
                    part[k][7][c] = h * (a.C[2 * n + nb] - a.C[2 * n + o]);
                }
            }
        }
        __syncthreads();
        if (sums)
            for (int q = 0; q < 8; ++q) {
                if (code[q][lane] == 0) continue;
                if (comp < 3) acc = fma(part[q][0][lane], part[q][1 + comp][lane], acc);
                else if (a.xf) acc = fma(part[q][4][lane], part[q][2 + comp][lane] - xP, acc);
                else acc += part[q][2 + comp][lane];
            }
        __syncthreads();
    }
    if (sums) (comp < 3 ? a.grad : a.U)[(size_t)(comp % 3) * n + cell] = acc * iv;
}

template <bool G, bool U>
__global__ void __launch_bounds__(256) k_grad_cells(GradArgs a)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= a.n) return;
    const int base = a.cf.ptr[c >> 5], w = (a.cf.ptr[(c >> 5) + 1] - base) >> 5, lane = c & 31;
    const size_t n = (size_t)a.n;
    const double iv = 1.0 / a.V[c];
    double xP0 = 0.0, xP1 = 0.0, xP2 = 0.0;
    if (U && a.xf) {
        xP0 = a.C[c];
        xP1 = a.C[n + c];
        xP2 = a.C[2 * n + c];
    }
    double g0 = 0.0, g1 = 0.0, g2 = 0.0, u0 = 0.0, u1 = 0.0, u2 = 0.0;
    constexpr int CH = 3;  // slots in flight
    for (int k0 = 0; k0 < w; k0 += CH) {
        int fo[CH];
        double4 rg[CH], ru[CH];
#pragma unroll
        for (int q = 0; q < CH; ++q) fo[q] = k0 + q < w ? a.cf.face[base + (k0 + q) * kSlice + lane] : 0;
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            const size_t f = (size_t)((fo[q] > 0 ? fo[q] : -fo[q]) - (fo[q] != 0));
            const double4 *rec = a.rec + f * ((int)G + (int)U);
            if (fo[q] != 0) {
                if (G) rg[q] = load_record(rec);
                if (U) ru[q] = load_record(rec + (int)G);
            }
        }
#pragma unroll
        for (int q = 0; q < CH; ++q) {
            if (fo[q] == 0) continue;
            if (G) {
                const double wt = fo[q] > 0 ? rg[q].w : 1.0 - rg[q].w;
                g0 = fma(wt, rg[q].x, g0);
                g1 = fma(wt, rg[q].y, g1);
                g2 = fma(wt, rg[q].z, g2);
            }
            if (U) {
                if (a.xf) {
                    const double ph = fo[q] > 0 ? ru[q].w : -ru[q].w;
                    u0 = fma(ph, ru[q].x - xP0, u0);
                    u1 = fma(ph, ru[q].y - xP1, u1);
                    u2 = fma(ph, ru[q].z - xP2, u2);
                } else {
                    u0 += ru[q].x;
                    u1 += ru[q].y;
                    u2 += ru[q].z;
                }
            }
        }
    }
    if (G) {
        a.grad[c] = g0 * iv;
        a.grad[n + c] = g1 * iv;
        a.grad[2 * n + c] = g2 * iv;
    }
    if (U) {
        a.U[c] = u0 * iv;
        a.U[n + c] = u1 * iv;
        a.U[2 * n + c] = u2 * iv;
    }
}

// Explicit over-relaxed non-orthogonal correction (Sec. 3), one thread per
// face: S_f = Delta_f + k_f with Delta_f = (S.S)/(S.d) d along the centre
// line (the implicit two-point part), and the k part from the gradient of
// the last p_d, interpolated to the face with the face-centre weight:
//     corr_f = rau_f k_f . (w_o G_own + (1 - w_o) G_nb),
// G = (1/rho) grad p_d (continuous across the interface by Eq. 8).  The face
// flux then reads phi*_f - corr_f - gamma_f (p_nb - p_own - J_f), so the cell
// sums take phi_eff = phi* - corr and sigma = phi_eff + gamma J.
// The gradient's face pass has left 1 - w_o = S.(x_f - x_o)/S.d in its record;
// (S.S)/(S.d) is the mesh's.
__global__ void __launch_bounds__(256) k_nonorth(NonorthArgs a)
{
    const int f = blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= a.F) return;
    const size_t n = (size_t)a.n, F = (size_t)a.F;
    const int o = a.owner[f], nb = a.neighbour[f];
    const double w_n = a.rec[f].w, w_o = 1.0 - w_n;
    double S[3], d[3], G[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        S[k] = a.Sf[k * F + f];
        d[k] = a.C[k * n + nb] - a.C[k * n + o];
        G[k] = fma(w_o, a.G[k * n + o], w_n * a.G[k * n + nb]);
    }
    const double over = a.c[f];  // (S.S)/(S.d)
    double kg = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) kg = fma(fma(-over, d[k], S[k]), G[k], kg);
    const double corr = (a.rau ? a.rau[f] : 1.0) * kg;
    const double pe = a.phi[f] - corr;
    a.corr[f] = corr;
    a.phi_eff[f] = pe;
    const double gam = a.gamma[f];
    a.gs[f] = make_double2(gam, pe + gam * a.jump[f]);
}

}  // namespace

cudaError_t launch_nonorth(const NonorthArgs &a, cudaStream_t s)
{
    if (a.F <= 0) return cudaSuccess;
    k_nonorth<<<(a.F + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

template <bool G, bool U>
static cudaError_t gradient(const GradArgs &a, cudaStream_t s)
{
    if (!a.rec) {
        k_grad_small<G, U><<<(a.n + 31) / 32, 256, 0, s>>>(a);
        return cudaGetLastError();
    }
    k_grad_faces<G, U><<<(a.F + 255) / 256, 256, 0, s>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_grad_cells<G, U><<<(a.n + 255) / 256, 256, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_gradient(const GradArgs &a, cudaStream_t s)
{
    if (a.n <= 0 || a.F <= 0) return cudaSuccess;
    if (a.grad && a.U) return gradient<true, true>(a, s);
    return a.grad ? gradient<true, false>(a, s) : gradient<false, true>(a, s);
}

}  // namespace gfm
