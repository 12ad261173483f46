"""The multigrid-preconditioned solve (every pinned system, unless
gfm_set_coarse(0)) against the CPU FP64 oracle and the Jacobi forms, at the
sizes where its levels can go wrong: one level only, a level of one node,
ragged slices, the hand-over from the grid to one CTA, wide rows of irregular
aggregates, disconnected meshes, tanks of very different depth in one batch.

Bars: true residual through the oracle's own matrix at the requested
tolerance (x1.05 for the rounding of the oracle's residual sum); p_d within
relative L2 1e-9 (FP64) and 1e-6 (mixed) of the oracle, as for every solve;
the iteration count, which multigrid keeps nearly independent of the mesh
size, below 80.
"""
import numpy as np
import pytest
import torch

import cases
import oracle

pytestmark = pytest.mark.gpu


def _g():
    import paper_1804_01130_gb300 as g
    return g


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _graded3d():
    rng = np.random.default_rng(6)
    m = cases.graded_mesh(*(np.concatenate([[0.0], np.cumsum(rng.uniform(0.02, 0.3, k))]) for k in (23, 17, 9)))
    alpha = np.clip((0.5 * m["C"][1].max() - m["C"][1]) / 0.1 + 0.5 + 0.3 * np.sin(3.0 * m["C"][0]), 0.0, 1.0)
    return cases._case_from(m, alpha, cases.random_face_flux(m, rng, two_d=False), "graded", (0, 16, 0))


def _wavy():
    m = cases.wavy_mesh(90, 47)
    alpha = np.clip((0.45 - m["C"][1]) * 47 + 0.5, 0.0, 1.0)
    return cases._case_from(m, alpha, cases.random_face_flux(m, np.random.default_rng(4), two_d=True), "wavy", (0, 46, 0))


CASES = {
    "two_cells": lambda: cases.column_case(ny=2, level=0.5173),
    "four_cells": lambda: cases.column_case(ny=4, level=0.5173),
    "five_cells": lambda: cases.column_case(ny=5, level=0.5173),
    "column_33": lambda: cases.column_case(ny=33, level=0.37),
    "column_257": lambda: cases.column_case(ny=257, level=0.41),
    "tank_37x19": lambda: cases.box_case(37, 19, 1, seed=8, nwaves=2),
    "tank_wide_cells": lambda: cases.box_case(24, 96, 1, seed=3, lx=6.0, ly=1.0),
    "tank_tall_cells": lambda: cases.box_case(160, 16, 1, seed=3, lx=1.0, ly=1.0),
    "tank_301x97": lambda: cases.box_case(301, 97, 1, seed=11, nwaves=3),
    "box_perm_noise": lambda: cases.box_case(21, 14, 11, seed=4, permute=True, alpha_noise=0.1),
    "drops_and_bubbles": lambda: cases.green_water_box(40, 24, 24, 7),
    "graded_3d": _graded3d,
    "wavy": _wavy,
}


@pytest.mark.parametrize("renumber", [0, 1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_multigrid_solve_matches_oracle(name, renumber):
    c = CASES[name]()
    p_ref, _, sy, _ = oracle.solve(c, direct=c.n <= 2048, rtol=1e-14)
    s = _g().GFM.from_case(c, renumber=renumber)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    for mode, bar in (("fp64", 1e-9), ("mixed", 1e-6)):
        p, _, info = s.solve(mode=mode, rtol=1e-12)
        pn = p.cpu().numpy()
        assert info.status == 0 and info.rel_res_l2 <= 1e-12 and info.iters < 80, (mode, info)
        assert np.linalg.norm(sy.b - oracle.spmv(sy, pn)) <= 1.05e-12 * np.linalg.norm(sy.b)
        assert _rel(pn, p_ref) <= bar
        again, _, info2 = s.solve(mode=mode, rtol=1e-12)
        assert torch.equal(again, p) and info2.iters == info.iters


def test_multigrid_agrees_with_the_jacobi_forms():
    """The same system through the path of gfm_set_coarse(0), with a face
    Rhie-Chow coefficient (every coefficient distinct) and a warm start."""
    c = cases.box_case(120, 50, 1, seed=5, nwaves=2)
    rau = np.random.default_rng(2).uniform(0.5, 2.0, c.F)
    out = []
    for vectors in (8, 0):
        s = _g().GFM.from_case(c)
        s.set_coarse(vectors)
        s.set_rau(rau)
        s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, 12.5)
        p, fl, i = s.solve(mode="fp64", rtol=1e-13, phi_corr=True)
        q, _, j = s.solve(mode="mixed", rtol=1e-12, p0=p * (1.0 + 1e-7))
        assert i.status == 0 and j.status == 0
        out.append((p.cpu().numpy(), q.cpu().numpy(), i.iters))
    assert _rel(out[0][0], out[1][0]) <= 1e-10 and _rel(out[0][1], out[1][0]) <= 1e-9
    assert out[0][2] < out[1][2] // 4


def test_multigrid_on_disconnected_parts():
    """A mesh of two parts that share no face: the pinned part is solved, the
    other one's source is compatible (zero flux, one phase)."""
    a, b = cases.structured_mesh(12, 9, 1, 1.0, 1.0, 0.1), cases.structured_mesh(7, 8, 1, 1.0, 1.0, 0.1)
    n = a["n"] + b["n"]
    own = np.concatenate([a["owner"], b["owner"] + a["n"]]).astype(np.int32)
    nb = np.concatenate([a["neighbour"], b["neighbour"] + a["n"]]).astype(np.int32)
    Sf, C = np.concatenate([a["Sf"], b["Sf"]], axis=1), np.concatenate([a["C"], b["C"]], axis=1)
    alpha = np.where(np.arange(n) < a["n"], np.clip((0.55 - C[1]) * 9 + 0.5, 0.0, 1.0), 1.0)
    phi = np.where(np.arange(own.size) < a["F"], 1e-3 * np.random.default_rng(1).normal(size=own.size), 0.0)
    s = _g().GFM(own, nb, Sf, C)
    s.assemble(torch.as_tensor(alpha), torch.as_tensor(phi), ref_cell=5)
    c = cases.Case("part", a["n"], a["F"], a["owner"], a["neighbour"], a["Sf"], a["C"], a["V"], a["xf"],
                   alpha=alpha[:a["n"]], phi=phi[:a["F"]], ref_cell=5)
    p_ref, _, _, _ = oracle.solve(c, direct=True)
    for mode in ("fp64", "mixed"):
        p, _, info = s.solve(mode=mode, rtol=1e-12)
        pn = p.cpu().numpy()
        assert info.status == 0
        assert _rel(pn[:a["n"]], p_ref) <= 1e-8
        assert np.abs(pn[a["n"]:]).max() <= 1e-8 * np.abs(p_ref).max()


@pytest.mark.parametrize("tuning", [None, (64, 1), (256, 2), (512, 1)])
def test_multigrid_batch_of_uneven_tanks(tuning):
    """Tanks from two cells to several levels, CTAs spanning many tanks and
    tanks spanning many CTAs."""
    tanks = [cases.column_case(ny=2, level=0.5173), cases.box_case(200, 70, 1, seed=1, nwaves=3),
             cases.column_case(ny=40, level=0.41), cases.box_case(5, 4, 1, seed=2), cases.box_case(97, 33, 1, seed=3)]
    tanks += [cases.box_case(6 + k, 5, 1, seed=20 + k) for k in range(9)]
    b = _g().GFMBatch(tanks)
    if tuning:
        b.set_tuning(*tuning)
    cat = lambda a: torch.as_tensor(np.concatenate([getattr(t, a) for t in tanks]))  # noqa: E731
    b.assemble(cat("alpha"), cat("phi"), [dict(rho_w=t.rho_w, rho_a=t.rho_a, g=t.g, ref_cell=t.ref_cell) for t in tanks])
    p, _, infos = b.solve(rtol=1e-12)
    pn, c0 = p.cpu().numpy(), 0
    for t, i in zip(tanks, infos):
        p_ref, _, _, _ = oracle.solve(t, direct=t.n <= 2048, rtol=1e-14)
        assert i.status == 0 and i.rel_res_l2 <= 1e-12 and i.iters < 80, i
        assert _rel(pn[c0:c0 + t.n], p_ref) <= 1e-6
        c0 += t.n


def test_multigrid_levels_follow_each_assembly():
    """Other alpha, other pinned cell, other rau on one handle: the coarse
    levels are those of the last assembly."""
    c = cases.box_case(80, 44, 1, seed=2, nwaves=2)
    d = cases.box_case(80, 44, 1, seed=9, nwaves=1, ka=0.15)
    s = _g().GFM.from_case(c)
    for k, (q, ref) in enumerate([(c, c.ref_cell), (d, 17), (c, c.n - 1), (d, 0)]):
        s.assemble(torch.as_tensor(q.alpha), torch.as_tensor(q.phi), q.rho_w, q.rho_a, q.g, ref)
        q.ref_cell = ref
        p_ref, _, _, _ = oracle.solve(q, direct=False, rtol=1e-14)
        p, _, info = s.solve(mode="fp64", rtol=1e-12)
        assert info.status == 0 and info.iters < 80 and _rel(p.cpu().numpy(), p_ref) <= 1e-9, (k, info)


@pytest.mark.parametrize("nx,ny", [(32, 32), (33, 32), (31, 32), (64, 64), (128, 64), (129, 64), (11, 3)])
def test_multigrid_small_levels_formed_in_one_launch(nx, ny):
    """Levels of at most 8 slices are formed by one CTA: the first coarse
    level at that size, one slice above and below, the second one there, and a
    mesh of small levels only.  Assembled twice: the second one's levels."""
    c = cases.box_case(nx, ny, 1, seed=6, nwaves=2)
    s = _g().GFM.from_case(c)
    args = (torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    s.assemble(torch.as_tensor(1.0 - c.alpha), *args)
    s.assemble(torch.as_tensor(c.alpha), *args)
    p_ref, _, _, _ = oracle.solve(c, direct=c.n <= 2048, rtol=1e-14)
    for mode, bar in (("fp64", 1e-9), ("mixed", 1e-6)):
        p, _, info = s.solve(mode=mode, rtol=1e-12)
        assert info.status == 0 and info.iters < 80 and _rel(p.cpu().numpy(), p_ref) <= bar, (mode, info)
