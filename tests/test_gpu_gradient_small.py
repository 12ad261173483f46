"""The gradient of small meshes, one launch of eight lanes a cell, and its line
to the two-pass form: meshes of one face to just above the line, a last slice
of one cell, cells of more faces than a chunk of eight, both outputs alone.

Bars as in test_gpu_gradient.py: 1e-12 of the largest terms that a cell's sum
can hold, |p| |S| / (V rho_a) and |phi| |x_f - x_P| / V."""
import numpy as np
import pytest
import torch

import cases
import oracle

pytestmark = pytest.mark.gpu


def _hub(n=67, seed=3):
    """Cells in a row, and two hubs of 24 and 17 faces: no mesh of a flow, but
    every face has its area, distance and centre."""
    rng = np.random.default_rng(seed)
    o = np.concatenate([np.arange(n - 1), np.zeros(23, int), np.full(15, 9)])
    v = np.concatenate([np.arange(1, n), np.arange(30, 53), np.arange(40, 55)])
    k = np.lexsort((v, o))
    o, v = o[k].astype(np.int32), v[k].astype(np.int32)
    C = rng.normal(size=(3, n))
    d = C[:, v] - C[:, o]
    S = d * rng.uniform(0.5, 2.0, o.size) + 0.05 * rng.normal(size=d.shape)
    xf = 0.5 * (C[:, o] + C[:, v]) + 0.05 * rng.normal(size=d.shape)
    return cases.Case("hub", n, o.size, o, v, S, C, rng.uniform(0.5, 2.0, n), xf, alpha=rng.uniform(0.0, 1.0, n),
                      phi=rng.normal(size=o.size), ref_cell=0)


CASES = {
    "one_face": lambda: cases.column_case(ny=2, level=0.5173),
    "column_33": lambda: cases.column_case(ny=33, level=0.37),  # a last slice of one cell
    "hub": _hub,
    "box_perm": lambda: cases.box_case(13, 11, 7, seed=4, permute=True, alpha_noise=0.1),
    "below_the_line": lambda: cases.box_case(150, 151, 1, seed=3, nwaves=2),  # 44,999 faces
    "above_the_line": lambda: cases.box_case(151, 151, 1, seed=3, nwaves=2),  # 45,300 faces
}


@pytest.mark.parametrize("use_xf", [False, True])
@pytest.mark.parametrize("name", sorted(CASES))
def test_gradient_of_small_meshes(name, use_xf):
    import paper_1804_01130_gb300 as g
    c = CASES[name]()
    s = g.GFM.from_case(c)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    p = np.random.default_rng(2).normal(size=c.n) * 1e3
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a))  # noqa: E731
    kw = dict(xf=t(c.xf) if use_xf else None)
    G, U = s.gradient(t(p), t(c.V), phi=t(c.phi), **kw)
    sv = np.max(np.linalg.norm(c.Sf, axis=0)) / np.min(c.V)
    reach = max(np.abs(c.xf - c.C[:, q]).max() for q in (c.owner, c.neighbour)) + np.abs(c.C[:, c.owner] - c.C[:, c.neighbour]).max()
    jump = np.abs(oracle.faces(c).jump).max()
    fac = 1.0
    if use_xf:  # the weights of faces whose centre lies off the line of the cells
        d = c.C[:, c.neighbour] - c.C[:, c.owner]
        fac += np.max(np.abs((c.Sf * (c.xf - c.C[:, c.owner])).sum(0) / (c.Sf * d).sum(0)))
    assert np.max(np.abs(G.cpu().numpy() - oracle.gradient(c, p, use_xf=use_xf))) <= 1e-12 * fac * (2e3 * 4 + jump) * sv / c.rho_a
    Ur = oracle.reconstruct(c, c.phi, use_xf=use_xf)
    assert np.max(np.abs(U.cpu().numpy() - Ur)) <= 1e-12 * np.abs(c.phi).max() * reach / np.min(c.V) * 8
    # each output alone: the same bits
    assert torch.equal(s.gradient(t(p), t(c.V), **kw)[0], G)
    assert torch.equal(s.gradient(t(p), t(c.V), phi=t(c.phi), want_grad=False, **kw)[1], U)
