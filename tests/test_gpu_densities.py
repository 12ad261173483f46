"""Assembly with densities that are awkward to divide by, bit for bit against
the oracle: off the interface gamma_f = c_f / rho is formed from 1 / rho and
an exact remainder, which has to round as the division does; where its
conditions fail (a significand of all ones, extreme exponents) it divides.
The gradient uses the same quotient."""
import math

import numpy as np
import pytest
import torch

import cases
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho_w,rho_a", [
    (998.2071, 1.2041), (3.0, 1.0 / 3.0), (1.0 + 2.0 ** -52, 1.0), (2.0 - 2.0 ** -52, 1.0 - 2.0 ** -53),
    (1e70, 1e-70), (7.0, 7.0), (math.pi * 1e3, math.e), (1025.0, 5e-324)])
def test_assembly_and_gradient_with_awkward_densities(rho_w, rho_a):
    import paper_1804_01130_gb300 as g
    c = cases.box_case(57, 31, 7, seed=13, nwaves=2, alpha_noise=0.2)
    c.rho_w, c.rho_a = rho_w, rho_a
    c.Sf = c.Sf * np.random.default_rng(3).uniform(0.5, 2.0, c.F)  # every c_f its own
    s = g.GFM.from_case(c)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    fc = oracle.faces(c)
    sy = oracle.assemble(c, fc)
    ex = {k: v.cpu().numpy() for k, v in s.export_system().items()}
    for k, ref in (("lambda", fc.lam), ("gamma", fc.gamma), ("jump", fc.jump), ("diag", sy.diag), ("b", sy.b)):
        assert np.array_equal(ex[k], ref, equal_nan=True), k  # rho_a = 5e-324: c/rho overflows on both sides
    if rho_a < 1e-60:
        return
    p = np.random.default_rng(1).normal(size=c.n)
    G, _ = s.gradient(torch.as_tensor(p), torch.as_tensor(c.V), xf=torch.as_tensor(c.xf))
    G_ref = oracle.gradient(c, p)
    # a cell's sum of six terms, each rounded a handful of times
    scale = np.max(np.abs(c.Sf)) / np.min(c.V) * (np.max(np.abs(p)) + np.max(np.abs(fc.jump))) / min(rho_a, rho_w)
    assert np.max(np.abs(G.cpu().numpy() - G_ref)) <= 64 * 2.0 ** -53 * scale
