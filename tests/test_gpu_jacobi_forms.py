"""The Jacobi kernels, which serve unpinned systems and gfm_set_coarse(0): the
compact and the full operator table, cached and streamed, the two-pass and the
fused form, single meshes and batches, each on handles that do run them (a
pinned system otherwise takes the multigrid kernel, which reads neither table
and has one form).  That they ran shows in the iteration count, several times
the multigrid solve's.

Bars, as for every solve: p_d within relative L2 1e-6 (mixed) of the CPU FP64
oracle; compact and full tables, and repeated solves, the same bits; the two
forms within 1e-7 of each other."""
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


def _assembled(c, coarse=0, renumber=1, form=1, ref=None):
    s = _g().GFM.from_case(c, renumber=renumber)
    s.set_coarse(coarse)
    s.set_tuning(form=form)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell if ref is None else ref,
               c.ref_value)
    return s


CASES = {
    "tank_40x24": lambda: cases.box_case(40, 24, 1, seed=3, ka=0.12),
    "box_24x16x12_perm": lambda: cases.box_case(24, 16, 12, seed=5, permute=True, alpha_noise=0.05),
    "tank_300x90": lambda: cases.box_case(300, 90, 1, seed=11, nwaves=3),
}


@pytest.mark.parametrize("stream", [False, True])
@pytest.mark.parametrize("renumber", [1, 2])
@pytest.mark.parametrize("name", sorted(CASES))
def test_compact_table_gives_the_full_ones_bits(name, renumber, stream):
    c = CASES[name]()
    mg = _assembled(c, 8, renumber).solve(mode="mixed", rtol=1e-10)[2].iters
    s, out = _assembled(c, 0, renumber), []
    assert s.table_info()["compact_usable"] and s.table_info()["compact_valid"]
    for compact in (True, False):
        s.set_table(compact=compact, force_stream=stream)
        p, _, info = s.solve(mode="mixed", rtol=1e-10)
        assert info.status == 0 and info.iters > 3 * mg, (compact, info, mg)
        out.append((p.clone(), info.iters))
    assert torch.equal(out[0][0], out[1][0]) and out[0][1] == out[1][1]
    p_ref = oracle.solve(c, direct=c.n <= 4096, rtol=1e-13)[0]
    assert _rel(out[0][0].cpu().numpy(), p_ref) <= 1e-6


def test_table_of_a_system_that_changes_its_solver():
    """Multigrid assemblies leave the compact table out: one in between must
    not leave an older system's table to a Jacobi solve."""
    c, d = cases.box_case(40, 24, 1, seed=3, ka=0.12), cases.box_case(40, 24, 1, seed=9, ka=0.05, nwaves=2)
    s, out = _g().GFM.from_case(c), []
    s.set_table(compact=True, force_stream=True)
    for q, vectors in ((c, 0), (d, 8), (d, 0)):
        s.set_coarse(vectors)
        s.assemble(torch.as_tensor(q.alpha), torch.as_tensor(q.phi), q.rho_w, q.rho_a, q.g, q.ref_cell, q.ref_value)
        assert s.table_info()["compact_valid"]  # it can hold the system, whichever solver runs
        out.append(s.solve(mode="mixed", rtol=1e-10)[0].cpu().numpy())
    for p, q in zip(out, (c, d, d)):
        assert _rel(p, oracle.solve(q, direct=True)[0]) <= 1e-6
    rau = torch.as_tensor(np.random.default_rng(4).uniform(0.5, 2.0, d.F))
    for vectors in (8, 0):
        s.set_coarse(vectors)
        s.set_rau(rau)
        s.assemble(torch.as_tensor(d.alpha), torch.as_tensor(d.phi), d.rho_w, d.rho_a, d.g, d.ref_cell, d.ref_value)
        assert not s.table_info()["compact_valid"]


@pytest.mark.parametrize("compact", [False, True])
@pytest.mark.parametrize("stream", [False, True])
def test_batch_of_tanks(stream, compact):
    tanks = cases.batch_cases(6, seed0=4300, nx_range=(40, 120), ny_range=(16, 48))
    cat = lambda a: torch.as_tensor(np.concatenate([getattr(t, a) for t in tanks]))  # noqa: E731
    phys = [dict(rho_w=t.rho_w, rho_a=t.rho_a, g=t.g, ref_cell=t.ref_cell, ref_value=t.ref_value) for t in tanks]
    out = []
    for vectors in (8, 0):
        b = _g().GFMBatch(tanks, renumber=1)
        b.set_coarse(vectors)
        b.set_table(compact=compact, force_stream=stream)
        b.assemble(cat("alpha"), cat("phi"), phys)
        assert vectors or b.table_info()["compact_valid"]
        p, _, infos = b.solve(rtol=1e-10)
        assert all(i.status == 0 for i in infos)
        again, _, _ = b.solve(rtol=1e-10)
        assert torch.equal(p, again)
        out.append((p.cpu().numpy(), infos))
    (_, mg), (pn, infos) = out
    c0 = 0
    for t, i, j in zip(tanks, infos, mg):
        assert i.iters > 3 * j.iters, (i, j)
        assert _rel(pn[c0:c0 + t.n], oracle.solve(t, rtol=1e-13, direct=False)[0]) <= 1e-6
        c0 += t.n


@pytest.mark.parametrize("name", sorted(CASES))
def test_fused_and_two_pass_form_agree(name):
    c = CASES[name]()
    mg = _assembled(c, 8).solve(mode="mixed", rtol=1e-10)[2].iters
    (p1, _, i1), (p2, _, i2) = (_assembled(c, form=f).solve(mode="mixed", rtol=1e-10) for f in (1, 2))
    assert i1.status == 0 and i2.status == 0 and min(i1.iters, i2.iters) > 3 * mg
    assert _rel(p2.cpu().numpy(), p1.cpu().numpy()) <= 1e-7


@pytest.mark.parametrize("form", [1, 2])
def test_warm_start_and_repetition(form):
    c = CASES["tank_300x90"]()
    s = _assembled(c, form=form)
    p, _, info = s.solve(mode="mixed", rtol=1e-10)
    p = p.clone()
    q, _, again = s.solve(mode="mixed", rtol=1e-10)
    assert torch.equal(p, q) and info.iters == again.iters
    p_ref = oracle.solve(c, direct=False, rtol=1e-14)[0]
    w, _, iw = s.solve(mode="mixed", rtol=1e-10, p0=torch.as_tensor(p_ref * (1.0 + 1e-6)))
    assert iw.status == 0 and iw.iters < info.iters and _rel(w.cpu().numpy(), p_ref) <= 1e-6


@pytest.mark.parametrize("form", [1, 2])
def test_adjoint(form):
    c = cases.make_case(1)
    w = np.where((np.abs(c.C[1] - 0.5) < 0.15) & (c.C[0] >= 0.5) & (c.C[0] <= 1.5), c.V, 0.0)
    dphi_ref, dalpha_ref, mu_ref, _ = oracle.adjoint(c, w, direct=c.n <= 2048, rtol=1e-14)
    s = _assembled(c, form=form)
    p, _, _ = s.solve(mode="fp64", rtol=1e-13)
    dphi, dalpha, mu, info = s.adjoint(p, torch.as_tensor(w), mode="mixed", rtol=1e-12)
    assert info.status == 0
    assert np.max(np.abs(mu.cpu().numpy() - mu_ref)) <= 1e-7 * np.abs(mu_ref).max()
    for got, ref in ((dphi, dphi_ref), (dalpha, dalpha_ref)):
        assert np.max(np.abs(got.cpu().numpy() - ref)) <= 1e-5 * np.abs(ref).max()


@pytest.mark.parametrize("form", [1, 2])
def test_time_step_equals_one_call_at_a_time(form):
    c = CASES["tank_300x90"]()
    dev, rng = torch.device("cuda"), np.random.default_rng(4)
    mesh = dict(xf=c.xf, Sf=c.Sf, spacing=(0.1, 0.1, 0.1), dims=c.dims)
    phis = np.stack([c.phi] + [c.phi + 1e-2 ** j * cases.random_face_flux(mesh, rng, two_d=True) for j in (1, 2)])
    phys = dict(rho_w=c.rho_w, rho_a=c.rho_a, g=c.g, ref_cell=c.ref_cell, ref_value=c.ref_value)
    s, ref = _assembled(c, form=form), _assembled(c, form=form)
    p, info = torch.zeros(c.n, dtype=torch.float64, device=dev), torch.zeros(12, dtype=torch.float64, device=dev)
    s.piso_step(torch.as_tensor(c.alpha, device=dev), torch.as_tensor(phis, device=dev), p, info,
                V=torch.as_tensor(c.V, device=dev), rtol=1e-10, **phys)
    torch.cuda.synchronize()
    infos, q = s.infos_of_step(info, 3), None
    assert all(i.status == 0 for i in infos)
    for j in range(3):
        ref.assemble(torch.as_tensor(c.alpha), torch.as_tensor(phis[j]), **phys)
        q, _, inf = ref.solve(mode="mixed", rtol=1e-10, p0=q)
        assert inf.iters == infos[j].iters
    assert torch.equal(p, q)
