"""The multigrid hierarchy's host set-up, on the CPU: each level's children
partition the finer level, every finer face between two aggregates belongs to
exactly one coarse face, the tables are symmetric, and a V-cycle over them
(restated in NumPy, with the kernels' weights) is symmetric positive definite
and preconditions CG to a count that hardly grows with the mesh."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

import cases

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <string>
#include "gfm_mg_setup.h"
#include "gfm_setup.h"
using namespace gfm;
struct H { HostTables t; std::vector<MgLevelHost> L; };
extern "C" {
void *mg_new(int n, int F, const int *o, const int *v, const double *S, const double *C, int ren) {
    H *h = new H; std::string e;
    if (!build_host_tables(n, F, o, v, C, ren, h->t, e)) { delete h; return nullptr; }
    h->L = build_mg_levels(n, h->t.n_pad, F, o, v, S, C, h->t.perm.data());
    return h;
}
int mg_n(void *p) { return (int)((H *)p)->L.size(); }
const int *mg_perm(void *p) { return ((H *)p)->t.perm.data(); }
void mg_dims(void *p, int l, int *d) { auto &q = ((H *)p)->L[l]; d[0] = q.n; d[1] = q.n_slices; d[2] = q.n_slots; d[3] = q.F; d[4] = (int)q.child.size(); d[5] = (int)q.mem.size(); }
const int *mg_int(void *p, int l, int w) { auto &q = ((H *)p)->L[l]; const std::vector<int32_t> *a[] = {&q.slice_ptr, &q.col, &q.face, &q.child_ptr, &q.child, &q.mem_ptr, &q.mem}; return a[w]->data(); }
const double *mg_scale(void *p, int l) { return ((H *)p)->L[l].scale.data(); }
void mg_del(void *p) { delete (H *)p; }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("mg")
    src = d / "shim.cpp"
    src.write_text(SHIM)
    csrc = os.path.join(ROOT, "paper_1804_01130_gb300", "csrc")
    out = str(d / "shim.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", csrc, str(src),
                    os.path.join(csrc, "gfm_mg_setup.cpp"), os.path.join(csrc, "gfm_setup.cpp"), "-o", out, "-lpthread"],
                   check=True)
    lb = ct.CDLL(out)
    lb.mg_new.restype = ct.c_void_p
    lb.mg_int.restype = lb.mg_perm.restype = ct.POINTER(ct.c_int)
    lb.mg_scale.restype = ct.POINTER(ct.c_double)
    return lb


def _hierarchy(lib, m, ren):
    arr = [np.ascontiguousarray(m[k], t) for k, t in (("owner", np.int32), ("neighbour", np.int32), ("Sf", float), ("C", float))]
    h = ct.c_void_p(lib.mg_new(m["n"], m["F"], *(ct.c_void_p(a.ctypes.data) for a in arr), ren))
    assert h.value
    levels = []
    for k in range(lib.mg_n(h)):
        d = (ct.c_int * 6)()
        lib.mg_dims(h, k, d)
        n, ns, nsl, F, nch, nm = d
        get = lambda w, c: np.ctypeslib.as_array(lib.mg_int(h, k, w), (max(c, 1),))[:c].copy()  # noqa: E731
        levels.append(dict(n=n, ns=ns, F=F, sp=get(0, ns + 1), col=get(1, nsl), face=get(2, nsl), cp=get(3, ns + 1),
                           child=get(4, nch), mp=get(5, F + 1), mem=get(6, nm),
                           scale=np.ctypeslib.as_array(lib.mg_scale(h, k), (max(F, 1),))[:F].copy()))
    perm = np.ctypeslib.as_array(lib.mg_perm(h), (m["n"],)).copy()
    lib.mg_del(h)
    return perm, levels


def _slots(ptr):
    """(slot, node) of every slot of a sliced-ELL list."""
    node = np.concatenate([np.tile(np.arange(32) + 32 * s, (ptr[s + 1] - ptr[s]) // 32) for s in range(len(ptr) - 1)])
    return node.astype(int)


def _check(m, perm, levels):
    n_f, o, v = m["n"], perm[m["owner"]], perm[m["neighbour"]]
    for L in levels:
        node = _slots(L["cp"])
        real = L["child"] >= 0
        assert np.array_equal(np.sort(L["child"][real]), np.arange(n_f))  # a partition (no padding cells here)
        agg = np.empty(n_f, int)
        agg[L["child"][real]] = node[real]
        assert agg.max() == L["n"] - 1 and np.all(np.bincount(agg) >= 1)
        # members: each finer face between two aggregates once, in ascending order
        cross = agg[o] != agg[v]
        assert np.array_equal(np.sort(L["mem"]), np.flatnonzero(cross))
        cf = np.repeat(np.arange(L["F"]), np.diff(L["mp"]))
        # the table: each face in the rows of its two aggregates
        row, f = _slots(L["sp"]), L["face"]
        assert np.array_equal(np.bincount(f[f > 0] - 1, minlength=L["F"]), np.full(L["F"], 2))
        lo, hi = np.full(L["F"], L["n"]), np.full(L["F"], -1)
        np.minimum.at(lo, f[f > 0] - 1, row[f > 0])
        np.maximum.at(hi, f[f > 0] - 1, row[f > 0])
        pair = np.sort(np.stack([agg[o], agg[v]]), axis=0)[:, L["mem"]]
        assert np.array_equal(pair, np.stack([lo[cf], hi[cf]]))
        other = L["col"][f > 0]
        assert np.array_equal(np.sort(np.stack([row[f > 0], other]), axis=0), np.stack([lo, hi])[:, f[f > 0] - 1])
        assert np.all(L["col"][f == 0] == row[f == 0]) and np.all(L["scale"] > 0)
        L["agg"], L["o"], L["v"], L["cf"] = agg, lo, hi, cf
        n_f, o, v = L["n"], lo, hi


def _vcycle(m, perm, levels, gamma, pin):
    """The preconditioner with the kernels' weights, on dense arrays in internal order."""
    w1, w2 = 0.56418, 1.69016
    ops = []
    o, v, n, g, p = perm[m["owner"]], perm[m["neighbour"]], m["n"], gamma, pin
    for k in range(len(levels) + 1):
        d = np.bincount(o, g, n) + np.bincount(v, g, n) + p
        ops.append((o, v, n, g, p, 1.0 / d))
        if k < len(levels):
            L = levels[k]
            g = L["scale"] * np.bincount(L["cf"], g[L["mem"]], L["F"])
            p = np.bincount(L["agg"], p, L["n"])
            o, v, n = L["o"], L["v"], L["n"]

    def mul(k, x):
        o, v, n, g, p, _ = ops[k]
        f = g * (x[o] - x[v])
        return np.bincount(o, f, n) - np.bincount(v, f, n) + p * x

    def cyc(k, b):
        di = ops[k][5]
        x = w1 * di * b
        x = x + w2 * di * (b - mul(k, x))
        if k + 1 < len(ops):
            a = levels[k]["agg"]
            x = x + cyc(k + 1, np.bincount(a, b - mul(k, x), levels[k]["n"]))[a]
        x = x + w2 * di * (b - mul(k, x))
        return x + w1 * di * (b - mul(k, x))
    return mul, cyc


MESHES = {
    "column_2": lambda: cases.structured_mesh(1, 2, 1, 0.1, 0.2, 0.1),
    "column_33": lambda: cases.structured_mesh(1, 33, 1, 0.1, 1.0, 0.1),
    "tank_64x32": lambda: cases.structured_mesh(64, 32, 1, 2.0, 1.0, 0.03),
    "tank_130x37": lambda: cases.structured_mesh(130, 37, 1, 16.0, 4.0, 0.1),
    "tall_cells": lambda: cases.structured_mesh(128, 16, 1, 1.0, 1.0, 0.1),
    "box_17x12x10": lambda: cases.structured_mesh(17, 12, 10, 2.0, 1.0, 1.0),
    "wavy": lambda: cases.wavy_mesh(40, 31),
    "box_permuted": lambda: cases.permute_mesh(cases.structured_mesh(16, 12, 9, 2.0, 1.0, 1.0),
                                               np.random.default_rng(0).permutation(16 * 12 * 9)),
}


@pytest.mark.parametrize("ren", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(MESHES))
def test_levels_and_vcycle(lib, name, ren):
    m = MESHES[name]()
    perm, levels = _hierarchy(lib, m, ren)
    _check(m, perm, levels)
    assert m["n"] <= 4 or levels[-1]["n"] <= 4
    # two phases with the densities' ratio, a pin, coefficients from the geometry
    d = m["C"][:, m["neighbour"]] - m["C"][:, m["owner"]]
    c = (m["Sf"] ** 2).sum(0) / (m["Sf"] * d).sum(0)
    wet = m["C"][1] < np.median(m["C"][1])
    both = wet[m["owner"]].astype(int) + wet[m["neighbour"]]
    gamma = c / np.array([1.0, 250.0, 1000.0])[both]
    pin = np.zeros(m["n"])
    pin[perm[0]] = gamma[(m["owner"] == 0) | (m["neighbour"] == 0)].sum()
    mul, cyc = _vcycle(m, perm, levels, gamma, pin)
    rng = np.random.default_rng(1)
    a, b = rng.normal(size=(2, m["n"]))
    assert abs(a @ cyc(0, b) - b @ cyc(0, a)) <= 1e-10 * abs(a @ cyc(0, a)) and a @ cyc(0, a) > 0
    r, it = mul(0, rng.normal(size=m["n"])), 0
    x, z = np.zeros(m["n"]), cyc(0, r)
    p, rz, r0 = z.copy(), r @ z, np.linalg.norm(r)
    while np.linalg.norm(r) > 1e-10 * r0 and it < 80:
        q = mul(0, p)
        al = rz / (p @ q)
        x += al * p
        r = r - al * q
        z = cyc(0, r)
        rz1 = r @ z
        p, rz, it = z + rz1 / rz * p, rz1, it + 1
    assert it < 60
