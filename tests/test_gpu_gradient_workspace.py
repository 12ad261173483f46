"""The gradient's workspace: on meshes of more than 262,144 faces allocated by
the first gradient, not by every handle, and that first call may be the one a
graph captures."""
import numpy as np
import pytest
import torch

import cases

pytestmark = pytest.mark.gpu


def _handle(c):
    import paper_1804_01130_gb300 as g
    s = g.GFM.from_case(c)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    return s


def _inputs(c):
    p = torch.as_tensor(np.random.default_rng(1).normal(size=c.n)).cuda()
    return dict(p=p, V=torch.as_tensor(c.V).cuda(), phi=torch.as_tensor(c.phi).cuda(), xf=torch.as_tensor(c.xf).cuda())


def test_first_gradient_allocates_its_workspace():
    """64 bytes a face; the driver hands out memory in blocks of 2 MiB."""
    c = cases.box_case(600, 400, 1, seed=2)
    s, a = _handle(c), _inputs(c)
    need = 64 * c.F
    out = torch.empty((6, c.n), dtype=torch.float64, device="cuda")  # the outputs' memory, in torch's cache
    del out
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    s.gradient(**a)
    torch.cuda.synchronize()
    first = torch.cuda.mem_get_info()[0]
    s.gradient(**a)
    torch.cuda.synchronize()
    assert before - first >= need - (2 << 20), (before - first, need)
    assert torch.cuda.mem_get_info()[0] == first


@pytest.mark.parametrize("call", ["gradient", "correction"])
def test_first_call_under_capture(call):
    """Gradient: the first call on the handle is the captured one.  Correction:
    its own workspace comes with an earlier call, the records with a gradient."""
    c = cases.box_case(400, 400, 1, seed=2)
    a = _inputs(c)
    if call == "gradient":
        ref = [t.clone() for t in _handle(c).gradient(**a)]
        s, st, graph = _handle(c), torch.cuda.Stream(), torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            out = s.gradient(**a, stream=st)
    else:
        args = (a["p"], a["V"])
        r = _handle(c)
        r.nonorth_correct(*args, xf=a["xf"])
        ref = [r.nonorth_correct(*args, xf=a["xf"], return_corr=True)]
        s, st, graph = _handle(c), torch.cuda.Stream(), torch.cuda.CUDAGraph()
        s.nonorth_correct(*args, xf=a["xf"])
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=st):
            out = [s.nonorth_correct(*args, xf=a["xf"], return_corr=True, stream=st)]
    graph.replay()
    torch.cuda.synchronize()
    for x, y in zip(out, ref):
        assert torch.equal(x, y)
