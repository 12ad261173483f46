// Host-side set-up of the multigrid preconditioner: aggregates, their graph
// and the geometric factors, from the mesh alone (built once per handle; the
// coefficients are formed on the device by every assembly).
//
// Each level merges nodes by passes of pairwise matching (two passes, groups
// of four, on 2D-like meshes; three, groups of eight, on 3D-like ones), the
// repeated pairwise aggregation of Notay (Electron. Trans. Numer. Anal. 37,
// 123-146, 2010) with a strength taken from the geometry.  A
// node is matched with its unmatched neighbour across the strongest face,
// the strength being the two-point coefficient |S|^2 / (S.d) of the merged
// face and the current centroids, so stretched cells are first merged along
// their short side (semi-coarsening) until the groups are about isotropic.
// Ties go to the lowest dominant axis of S, which on structured meshes gives
// rectangular groups in every cell order that sweeps the mesh (the caller's,
// RCM, Morton).  A node left without an unmatched neighbour joins the pair
// behind its strongest face.
//
// A coarse face gets the factor |sum S|^2 / (sum S . d_coarse) over the sum
// of its finer faces' |S|^2 / (S.d): on a uniform mesh 1/2 per level.  The
// plain Galerkin sum of the faces' coefficients overestimates the coarse
// energy by about two, since the groups' interpolation is piecewise constant;
// scaled this way the coarse operator is the two-point operator of the
// merged cells.
#include <algorithm>
#include <cmath>
#include <exception>
#include <numeric>
#include <thread>

#include "gfm_mg_setup.h"
#include "gfm_setup.h"

namespace gfm {

namespace {

struct Graph {
    int n = 0;
    std::vector<int32_t> o, v;       // faces
    std::vector<double> S[3];        // area vectors, o -> v
    std::vector<double> P[3], w;     // node centroids and weights
    int F() const { return (int)o.size(); }
};

struct Adj {
    std::vector<int32_t> ptr, nbr, face;
};

// fn(lo, hi) over [0, n) in stretches on the host's cores (small ranges inline).
template <typename Fn>
void parallel_ranges(int n, Fn fn)
{
    const int most = (int)std::min<unsigned>(16u, std::max(1u, std::thread::hardware_concurrency()));
    const int nt = std::min(most, n / 65536);
    if (nt < 2) {
        fn(0, n);
        return;
    }
    std::vector<std::thread> th;
    th.reserve((size_t)nt);
    int t = 0;
    try {
        for (; t < nt; ++t) th.emplace_back(fn, (int)((long long)n * t / nt), (int)((long long)n * (t + 1) / nt));
    } catch (const std::exception &) {  // no thread (or memory for one) to be had: the rest here
        fn((int)((long long)n * t / nt), n);
    }
    for (auto &q : th) q.join();
}

double strength(const Graph &g, int f)
{
    double ss = 0.0, sd = 0.0;
    const int o = g.o[(size_t)f], v = g.v[(size_t)f];
    for (int k = 0; k < 3; ++k) {
        const double s = g.S[k][(size_t)f];
        ss += s * s;
        sd += s * (g.P[k][(size_t)v] - g.P[k][(size_t)o]);
    }
    sd = std::fabs(sd);
    return sd > 0.0 ? ss / sd : 0.0;
}

void build_adj(const Graph &g, Adj &a)
{
    const int F = g.F();
    a.ptr.assign((size_t)g.n + 1, 0);
    for (int f = 0; f < F; ++f) {
        a.ptr[(size_t)g.o[(size_t)f] + 1]++;
        a.ptr[(size_t)g.v[(size_t)f] + 1]++;
    }
    for (int i = 0; i < g.n; ++i) a.ptr[(size_t)i + 1] += a.ptr[(size_t)i];
    a.nbr.resize(2 * (size_t)F);
    a.face.resize(2 * (size_t)F);
    std::vector<int32_t> pos(a.ptr.begin(), a.ptr.end() - 1);
    for (int f = 0; f < F; ++f) {
        const int32_t o = g.o[(size_t)f], v = g.v[(size_t)f];
        a.nbr[(size_t)pos[o]] = v;
        a.face[(size_t)pos[o]++] = f;
        a.nbr[(size_t)pos[v]] = o;
        a.face[(size_t)pos[v]++] = f;
    }
}

// One matching pass in node order; grp[i] = group of node i, numbered in the
// order the groups are opened.  Returns the number of groups.
int match_pass(const Graph &g, const Adj &a, const std::vector<float> &c, const std::vector<uint8_t> &axis,
               std::vector<int32_t> &grp)
{
    constexpr float kTie = 0.05f;  // strengths within 5% count as equal
    grp.assign((size_t)g.n, -1);
    std::vector<uint8_t> size;
    size.reserve((size_t)g.n / 2 + 1);
    int ng = 0;
    for (int i = 0; i < g.n; ++i) {
        if (grp[(size_t)i] >= 0) continue;
        int bf = -1, bj = -1;
        for (int32_t e = a.ptr[(size_t)i]; e < a.ptr[(size_t)i + 1]; ++e) {
            const int j = a.nbr[(size_t)e], f = a.face[(size_t)e];
            if (grp[(size_t)j] >= 0) continue;
            if (bf < 0 || c[(size_t)f] > c[(size_t)bf] * (1.0f + kTie)) {
                bf = f;
                bj = j;
            } else if (c[(size_t)f] >= c[(size_t)bf] * (1.0f - kTie)) {
                if (axis[(size_t)f] < axis[(size_t)bf] || (axis[(size_t)f] == axis[(size_t)bf] && j < bj)) {
                    bf = f;
                    bj = j;
                }
            }
        }
        if (bj >= 0) {
            grp[(size_t)i] = grp[(size_t)bj] = ng++;
            size.push_back(2);
            continue;
        }
        int best = -1, bg = -1;
        for (int32_t e = a.ptr[(size_t)i]; e < a.ptr[(size_t)i + 1]; ++e) {
            const int q = grp[(size_t)a.nbr[(size_t)e]], f = a.face[(size_t)e];
            if (q < 0 || size[(size_t)q] > 2) continue;
            if (best < 0 || c[(size_t)f] > c[(size_t)best]) {
                best = f;
                bg = q;
            }
        }
        if (bg >= 0) {
            grp[(size_t)i] = bg;
            size[(size_t)bg]++;
        } else {
            grp[(size_t)i] = ng++;
            size.push_back(1);
        }
    }
    return ng;
}

// The graph of the groups; fmap[f] = coarse face of finer face f, -1 inside a group.
Graph merge(const Graph &g, const Adj &a, const std::vector<int32_t> &grp, int ng, std::vector<int32_t> &fmap)
{
    Graph c;
    c.n = ng;
    for (int k = 0; k < 3; ++k) c.P[k].assign((size_t)ng, 0.0);
    c.w.assign((size_t)ng, 0.0);
    std::vector<int32_t> ptr((size_t)ng + 1, 0), mem((size_t)g.n);
    for (int i = 0; i < g.n; ++i) {
        const int q = grp[(size_t)i];
        ptr[(size_t)q + 1]++;
        c.w[(size_t)q] += g.w[(size_t)i];
        for (int k = 0; k < 3; ++k) c.P[k][(size_t)q] += g.w[(size_t)i] * g.P[k][(size_t)i];
    }
    for (int q = 0; q < ng; ++q) {
        ptr[(size_t)q + 1] += ptr[(size_t)q];
        for (int k = 0; k < 3; ++k) c.P[k][(size_t)q] /= c.w[(size_t)q];
    }
    std::vector<int32_t> pos(ptr.begin(), ptr.end() - 1);
    for (int i = 0; i < g.n; ++i) mem[(size_t)pos[(size_t)grp[(size_t)i]]++] = i;
    fmap.assign((size_t)g.F(), -1);
    const size_t guess = (size_t)g.F() * 6 / 10 + 16;
    c.o.reserve(guess);
    c.v.reserve(guess);
    for (int k = 0; k < 3; ++k) c.S[k].reserve(guess);
    std::vector<int32_t> mark((size_t)ng, -1);  // face to each neighbour of the current group
    for (int q = 0; q < ng; ++q) {
        const int first = (int)c.o.size();
        for (int32_t m = ptr[(size_t)q]; m < ptr[(size_t)q + 1]; ++m) {
            const int i = mem[(size_t)m];
            for (int32_t e = a.ptr[(size_t)i]; e < a.ptr[(size_t)i + 1]; ++e) {
                const int r = grp[(size_t)a.nbr[(size_t)e]], f = a.face[(size_t)e];
                if (r <= q) continue;  // inside the group, or listed by the lower group
                int cf = mark[(size_t)r];
                if (cf < first) {
                    cf = mark[(size_t)r] = (int)c.o.size();
                    c.o.push_back(q);
                    c.v.push_back(r);
                    for (int k = 0; k < 3; ++k) c.S[k].push_back(0.0);
                }
                fmap[(size_t)f] = cf;
                const double sg = g.o[(size_t)f] == i ? 1.0 : -1.0;
                for (int k = 0; k < 3; ++k) c.S[k][(size_t)cf] += sg * g.S[k][(size_t)f];
            }
        }
    }
    return c;
}

// Counting sort of items 0..m-1 by key (-1 dropped): ptr [nk + 1], list ascending in each key.
void group_by(const std::vector<int32_t> &key, int nk, std::vector<int32_t> &ptr, std::vector<int32_t> &list)
{
    ptr.assign((size_t)nk + 1, 0);
    for (int32_t k : key)
        if (k >= 0) ptr[(size_t)k + 1]++;
    for (int k = 0; k < nk; ++k) ptr[(size_t)k + 1] += ptr[(size_t)k];
    list.resize((size_t)ptr[(size_t)nk]);
    std::vector<int32_t> pos(ptr.begin(), ptr.end() - 1);
    for (size_t i = 0; i < key.size(); ++i)
        if (key[i] >= 0) list[(size_t)pos[(size_t)key[i]]++] = (int32_t)i;
}

// Sliced-ELL form of per-node lists: slots of node i of slice s at ptr[s] + k * 32 + lane.
template <typename Fn>
int to_sell(int n, int n_slices, const std::vector<int32_t> &cnt_ptr, std::vector<int32_t> &slice_ptr, Fn fill)
{
    slice_ptr.assign((size_t)n_slices + 1, 0);
    int maxw = 0;
    for (int s = 0; s < n_slices; ++s) {
        int w = 0;
        for (int i = s * kSliceH; i < std::min(n, (s + 1) * kSliceH); ++i)
            w = std::max(w, cnt_ptr[(size_t)i + 1] - cnt_ptr[(size_t)i]);
        maxw = std::max(maxw, w);
        slice_ptr[(size_t)s + 1] = slice_ptr[(size_t)s] + w * kSliceH;
    }
    for (int s = 0; s < n_slices; ++s) {
        const int base = slice_ptr[(size_t)s], w = (slice_ptr[(size_t)s + 1] - base) / kSliceH;
        for (int l = 0; l < kSliceH; ++l) {
            const int i = s * kSliceH + l;
            const int m = i < n ? cnt_ptr[(size_t)i + 1] - cnt_ptr[(size_t)i] : 0;
            for (int k = 0; k < w; ++k) fill(base + k * kSliceH + l, i, k < m ? cnt_ptr[(size_t)i] + k : -1);
        }
    }
    return maxw;
}

}  // namespace

std::vector<MgLevelHost> build_mg_levels(int n, int n_pad, int F, const int32_t *owner, const int32_t *nb,
                                         const double *Sf, const double *C, const int32_t *perm,
                                         const int32_t *slot_face, int n_slots)
{
    std::vector<MgLevelHost> levels;
    // the mesh, its cells numbered in internal order without the padding cells
    std::vector<int32_t> real((size_t)n_pad, -1), cell;  // internal -> dense and back
    for (int i = 0; i < n; ++i) real[(size_t)perm[i]] = 1;
    cell.reserve((size_t)n);
    for (int i = 0; i < n_pad; ++i)
        if (real[(size_t)i] > 0) {
            real[(size_t)i] = (int32_t)cell.size();
            cell.push_back(i);
        }
    // faces sorted by their lower cell, so that every pass over them walks the
    // cells in order whatever the caller's order: at[q] = caller face of face q
    std::vector<int32_t> fo((size_t)F), fv((size_t)F), low((size_t)F), ptr, at;
    parallel_ranges(F, [&](int lo, int hi) {
        for (int f = lo; f < hi; ++f) {
            fo[(size_t)f] = real[(size_t)perm[owner[f]]];
            fv[(size_t)f] = real[(size_t)perm[nb[f]]];
            low[(size_t)f] = std::min(fo[(size_t)f], fv[(size_t)f]);
        }
    });
    group_by(low, n, ptr, at);
    Graph g;
    g.n = n;
    g.o.resize((size_t)F);
    g.v.resize((size_t)F);
    for (int k = 0; k < 3; ++k) {
        g.S[k].resize((size_t)F);
        g.P[k].resize((size_t)n);
    }
    parallel_ranges(F, [&](int lo, int hi) {
        for (int q = lo; q < hi; ++q) {
            const size_t f = (size_t)at[(size_t)q];
            g.o[(size_t)q] = fo[f];
            g.v[(size_t)q] = fv[f];
            for (int k = 0; k < 3; ++k) g.S[k][(size_t)q] = Sf[(size_t)k * F + f];
        }
    });
    parallel_ranges(n, [&](int lo, int hi) {
        for (int i = lo; i < hi; ++i)
            for (int k = 0; k < 3; ++k) g.P[k][(size_t)real[(size_t)perm[i]]] = C[(size_t)k * n + i];
    });
    g.w.assign((size_t)n, 1.0);
    const int passes = (double)F > 2.3 * (double)n ? 3 : 2;
    while (g.n > kMgCoarsest && (int)levels.size() + 1 < kMgMaxLevels) {
        const int n0 = g.n, F0 = g.F();
        std::vector<int32_t> grp, fm;  // finer node -> group, finer face -> coarse face
        std::vector<double> c0((size_t)F0);
        parallel_ranges(F0, [&](int lo, int hi) {
            for (int f = lo; f < hi; ++f) c0[(size_t)f] = strength(g, f);
        });
        Graph cur;
        const Graph *gp = &g;
        for (int p = 0; p < passes; ++p) {
            const int Fp = gp->F();
            Adj adj;
            build_adj(*gp, adj);
            std::vector<float> c((size_t)Fp);
            std::vector<uint8_t> axis((size_t)Fp);
            parallel_ranges(Fp, [&](int lo, int hi) {
                for (int f = lo; f < hi; ++f) {
                    c[(size_t)f] = (float)(p == 0 ? c0[(size_t)f] : strength(*gp, f));
                    double m = -1.0;
                    for (int k = 0; k < 3; ++k) {
                        const double s = std::fabs(gp->S[k][(size_t)f]);
                        if (s > m * 1.0001) {
                            m = s;
                            axis[(size_t)f] = (uint8_t)k;
                        }
                    }
                }
            });
            std::vector<int32_t> pg, pf;
            const int ng = match_pass(*gp, adj, c, axis, pg);
            Graph nx = merge(*gp, adj, pg, ng, pf);
            if (p == 0) {
                grp.swap(pg);
                fm.swap(pf);
            } else {
                for (auto &q : grp) q = pg[(size_t)q];
                for (auto &f : fm)
                    if (f >= 0) f = pf[(size_t)f];
            }
            cur = std::move(nx);
            gp = &cur;
        }
        if (cur.n > 0.8 * n0) break;  // nothing left to merge
        MgLevelHost L;
        L.n = cur.n;
        L.F = cur.F();
        L.n_slices = (L.n + kSliceH - 1) / kSliceH;
        L.n_pad = L.n_slices * kSliceH;
        group_by(fm, L.F, L.mem_ptr, L.mem);
        L.scale.resize((size_t)L.F);
        for (int f = 0; f < L.F; ++f) {
            double s = 0.0;
            for (int32_t m = L.mem_ptr[(size_t)f]; m < L.mem_ptr[(size_t)f + 1]; ++m) s += c0[(size_t)L.mem[(size_t)m]];
            const double r = s > 0.0 ? strength(cur, f) / s : 0.5;
            L.scale[(size_t)f] = std::min(2.0, std::max(0.05, r));
        }
        if (levels.empty()) {  // members in the caller's face numbers, or as slots
            std::vector<int32_t> slot;
            if (slot_face) {
                slot.resize((size_t)F);
                parallel_ranges(n_slots, [&](int lo, int hi) {
                    for (int q = lo; q < hi; ++q)
                        if (slot_face[q] > 0) slot[(size_t)slot_face[q] - 1] = q;
                });
            }
            parallel_ranges((int)L.mem.size(), [&](int lo, int hi) {
                for (int q = lo; q < hi; ++q) {
                    const int32_t f = at[(size_t)L.mem[(size_t)q]];
                    L.mem[(size_t)q] = slot_face ? slot[(size_t)f] : f;
                }
            });
        }
        Adj adj;
        build_adj(cur, adj);
        L.max_width = to_sell(L.n, L.n_slices, adj.ptr, L.slice_ptr, [&](int slot, int i, int e) {
            if ((size_t)slot >= L.col.size()) {
                L.col.resize((size_t)L.slice_ptr[(size_t)L.n_slices]);
                L.face.resize((size_t)L.slice_ptr[(size_t)L.n_slices]);
            }
            L.col[(size_t)slot] = e >= 0 ? adj.nbr[(size_t)e] : i;
            L.face[(size_t)slot] = e >= 0 ? adj.face[(size_t)e] + 1 : 0;
        });
        L.n_slots = L.slice_ptr[(size_t)L.n_slices];
        std::vector<int32_t> cptr, clist;
        group_by(grp, L.n, cptr, clist);
        L.max_child = to_sell(L.n, L.n_slices, cptr, L.child_ptr, [&](int slot, int, int e) {
            if ((size_t)slot >= L.child.size()) L.child.resize((size_t)L.child_ptr[(size_t)L.n_slices]);
            const int32_t ch = e >= 0 ? clist[(size_t)e] : -1;
            // children of the first coarse level are cells: back to internal numbers
            L.child[(size_t)slot] = (ch >= 0 && levels.empty()) ? cell[(size_t)ch] : ch;
        });
        levels.push_back(std::move(L));
        g = std::move(cur);
    }
    return levels;
}

}  // namespace gfm
