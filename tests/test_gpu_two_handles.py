"""Two handles of different size at once: each has its own host thread (a handle
is one thread's, the library is not), and a captured solve of one is replayed
after the other has solved.  The kernels' shared-memory limit
belongs to the function, not to a handle: what one handle plans must not take
it from the other.  Results are those of each handle alone, bit for bit."""
import threading

import pytest
import torch

import cases

pytestmark = pytest.mark.gpu


def _g():
    import paper_1804_01130_gb300 as g
    return g


def _handle(c, coarse):
    s = _g().GFM.from_case(c)
    s.set_coarse(coarse)
    s.assemble(torch.as_tensor(c.alpha), torch.as_tensor(c.phi), c.rho_w, c.rho_a, c.g, c.ref_cell, c.ref_value)
    return s


# a table held in shared memory (the most of it), a tail alone, a few levels
SIZES = [(400, 160), (40, 24)]


@pytest.mark.parametrize("coarse", [8, 0])
@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_two_threads_solve_on_one_stream(mode, coarse):
    hs = [_handle(cases.box_case(nx, ny, 1, seed=3, nwaves=2), coarse) for nx, ny in SIZES]
    alone = [h.solve(mode=mode, rtol=1e-6)[0].clone() for h in hs]
    torch.cuda.synchronize()
    failures, gate, s = [], threading.Barrier(2), torch.cuda.Stream()

    def work(h, p_alone, n):
        try:
            out = torch.empty_like(p_alone)
            gate.wait()
            with torch.cuda.stream(s):
                for k in range(n):
                    h.solve(mode=mode, rtol=1e-6, info_on_device=True, out=out, stream=s)
                    if k % 16 == 15:
                        s.synchronize()
            s.synchronize()
            if not torch.equal(out, p_alone):
                failures.append("another solution")
        except Exception as e:  # noqa: BLE001 - reported by the test
            failures.append(repr(e))

    ts = [threading.Thread(target=work, args=(h, a, n)) for h, a, n in zip(hs, alone, (200, 400))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failures, failures[:3]


@pytest.mark.parametrize("mode", ["mixed", "fp64"])
def test_a_captured_solve_survives_another_handle(mode):
    big, small = (_handle(cases.box_case(nx, ny, 1, seed=3, nwaves=2), 8) for nx, ny in SIZES)
    alone = big.solve(mode=mode, rtol=1e-6)[0].clone()
    s, out, graph = torch.cuda.Stream(), torch.empty_like(alone), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        big.solve(mode=mode, rtol=1e-6, info_on_device=True, out=out, stream=s)
        small.solve(mode=mode, rtol=1e-6, info_on_device=True, stream=s)
    small.solve(mode=mode, rtol=1e-6)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, alone)
