"""Multigrid solves whose tolerance lies near the rounding floor: the
adjoint of a two-gauge pressure difference (its right-hand side's residual
cannot be brought below about 6e-13 at 256x128) on many free surfaces, and
long shallow or tall tanks.  Every solve ends, and with status 0 wherever the
Jacobi form (gfm_set_coarse(0)) gets there.

Bars: an ordinary tank takes 25 to 35 V-cycles, re-checks at the floor
included, so 100 is far above; the longest tanks here (length / depth 160)
take a few hundred, so 400."""
import numpy as np
import pytest
import torch

import cases

pytestmark = pytest.mark.gpu

NOT_CONVERGED = 4


def _g():
    import paper_1804_01130_gb300 as g
    return g


def _probe(c, lx, ly):
    """Weights of a pressure difference between two gauges under water."""
    w = [c.V * np.exp(-((c.C[0] - x * lx) ** 2 + (c.C[1] - 0.25 * ly) ** 2) / (0.1 * ly) ** 2) for x in (0.3, 0.7)]
    return torch.as_tensor(w[0] / w[0].sum() - w[1] / w[1].sum())


def _assemble(s, c):
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)


def test_adjoint_ends_at_the_floor_on_many_surfaces():
    s, bad = None, []
    for k in range(64):
        c = cases.box_case(256, 128, 1, seed=k, nwaves=2, lx=4.0, ly=2.0, ka=0.06 + 0.001 * k)
        s = s or _g().GFM.from_case(c)
        _assemble(s, c)
        p, _, i = s.solve(mode="fp64", rtol=1e-12, max_iters=2000, raise_on_error=False)
        _, _, _, j = s.adjoint(p, _probe(c, 4.0, 2.0), rtol=1e-12, max_iters=2000, raise_on_error=False)
        bad += [(k, q) for q in (i, j) if q.status != 0 or q.iters >= 100 or q.rel_res_l2 > 1e-12]
    assert not bad, bad


@pytest.mark.parametrize("aspect", [0.3, 1.0, 4.0])
@pytest.mark.parametrize("nx,ny", [(843, 21), (497, 54), (913, 25), (1344, 21), (44, 438), (115, 212)])
def test_long_and_tall_tanks_end(nx, ny, aspect):
    """aspect: width of a cell over its height."""
    lx, ly = 2.0 * nx / ny * aspect, 2.0
    c = cases.box_case(nx, ny, 1, seed=7, nwaves=1, lx=lx, ly=ly, ka=0.05)
    w, out = _probe(c, lx, ly), []
    for vectors in (8, 0):
        s = _g().GFM.from_case(c)
        s.set_coarse(vectors)
        _assemble(s, c)
        p, _, i = s.solve(mode="fp64", rtol=1e-12, max_iters=40_000 if vectors == 0 else 2000, raise_on_error=False)
        _, _, _, j = s.adjoint(p, w, rtol=1e-12, max_iters=40_000 if vectors == 0 else 2000, raise_on_error=False)
        out.append((i, j))
    for mg, jacobi in zip(*out):
        if jacobi.status == 0:
            assert mg.status == 0 and mg.rel_res_l2 <= 1e-12 and mg.iters < 400, (mg, jacobi)
        else:
            assert mg.status in (0, NOT_CONVERGED) and mg.iters < 2000, (mg, jacobi)


def test_mixed_adjoint_just_above_the_floor():
    """24x18 cells, a band across the surface: the rounding of x leaves about
    1.0e-13, the Jacobi form ends at 1.6e-13; asked for 1e-13."""
    c = cases.box_case(24, 18, 1, seed=3, nwaves=2, lx=2.0, ly=1.0, ka=0.05)
    s = _g().GFM.from_case(c)
    _assemble(s, c)
    p, _, _ = s.solve(mode="mixed", rtol=1e-13)
    w = torch.as_tensor(np.where(np.abs(c.C[1] - 0.5) < 0.15, c.V, 0.0))
    _, _, _, i = s.adjoint(p, w, mode="mixed", rtol=1e-13, raise_on_error=False)
    assert i.status == 0 and i.rel_res_l2 <= 1e-13 and i.iters < 100, i
