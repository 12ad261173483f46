"""The FP64 multigrid solve's rules at a residual replacement, restated in
NumPy over the library's own hierarchy: r becomes the true residual, the
directions start anew, the steps since are folded into x at once, and a claim
that was refuted halves the next one's target.  Near the rounding floor the
true residual is mostly the rounding of x; a direction kept across the
replacement makes the residual grow there."""
import math

import numpy as np
import pytest
import scipy.sparse as sp

import cases
import oracle
from test_mg_setup import _check, _hierarchy, _vcycle, lib  # noqa: F401


def _solve(A, mul, cyc, b, rtol=1e-12, most=200):
    bn, x, e, r = np.linalg.norm(b), np.zeros_like(b), np.zeros_like(b), b.copy()
    p = s = None
    gam, best, stall, it, target = 1.0, math.inf, 0, 0, 0.81
    while it < most:
        rr = r @ r
        if math.sqrt(rr) <= rtol * bn:
            return it, math.sqrt(rr) / bn
        stall = 0 if rr < 0.25 * best else stall + 1
        best = min(best, rr)
        if stall > 3:
            break
        fresh = True
        while it < most:
            z = cyc(0, r)
            g = r @ z
            be = 0.0 if fresh else g / gam
            s, p = (A @ z, z) if fresh else (A @ z + be * s, z + be * p)
            fresh, gam, al = False, g, g / (p @ s)
            e, r, it = e + al * p, r - al * s, it + 1
            if r @ r <= target * (rtol * bn) ** 2:
                break
        target *= 0.25
        x, e = x + e, np.zeros_like(b)
        r = b - mul(0, x)
    return it, math.sqrt(r @ r) / bn


def _adjoint_system(lib, ka):  # noqa: F811
    c = cases.box_case(256, 128, 1, seed=3, nwaves=2, lx=4.0, ly=2.0, ka=ka)
    m = dict(n=c.n, F=c.F, owner=c.owner, neighbour=c.neighbour, Sf=c.Sf, C=c.C)
    perm, levels = _hierarchy(lib, m, 1)
    _check(m, perm, levels)
    gamma = oracle.faces(c).gamma
    pin = np.zeros(c.n)
    pin[perm[c.ref_cell]] = gamma[(c.owner == c.ref_cell) | (c.neighbour == c.ref_cell)].sum()
    w = [c.V * np.exp(-((c.C[0] - x * 4.0) ** 2 + (c.C[1] - 0.5) ** 2) / 0.04) for x in (0.3, 0.7)]
    b = np.zeros(c.n)
    b[perm] = w[0] / w[0].sum() - w[1] / w[1].sum()
    o, v = perm[c.owner], perm[c.neighbour]
    diag = np.bincount(o, gamma, c.n) + np.bincount(v, gamma, c.n) + pin
    # the direction's A z in diagonal form, the true residual in difference form
    i = np.arange(c.n)
    A = sp.csr_matrix((np.concatenate([diag, -gamma, -gamma]), (np.concatenate([i, o, v]), np.concatenate([i, v, o]))))
    return (A, *_vcycle(m, perm, levels, gamma, pin), b)


@pytest.mark.parametrize("ka", [0.08, 0.1, 0.116])
def test_directions_start_anew_at_a_replacement(lib, ka):  # noqa: F811
    system = _adjoint_system(lib, ka)
    it, rel = _solve(*system)
    assert rel <= 1e-12 and it < 60, (it, rel)
