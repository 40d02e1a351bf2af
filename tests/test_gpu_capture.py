"""FP64 Q_tm and CUDA graphs: its fixed-point scratch leaves the scratch of a
graph captured around another operator alone, and a call first made inside a
capture (no fixed-point scratch yet) is captured all the same."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


@pytest.mark.parametrize("dims", [(8, 8, 8, 8), (16, 16, 16, 16)])   # split over warps, and with a converted input
def test_capture_before_the_first_qtm(dims):
    from paper_1311_4521_gb300 import tmhop
    vh = int(np.prod(dims)) // 2
    U, psi, chi = F.gauge_field(dims, 950, "random"), F.gaussian_spinor(vh, 950, 1), F.gaussian_spinor(vh, 950, 2)
    c = tmhop.Context(0)
    g = c.gauge(dims, U, "f64", 18)
    a, b = c.pack(psi, "f64"), c.pack(chi, "f64")
    outs, one = [c.empty(vh, "f64"), c.empty(vh, "f64")], c.empty(vh, "f64")
    c.Qnd(g, outs, [a, b], 0.16, 0.01, 0.02)   # makes the scratch of the other operators
    want = [c.unpack(o, vh, "f64").cpu().numpy() for o in outs]
    nd, qtm = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(nd):
        c.Qnd(g, outs, [a, b], 0.16, 0.01, 0.02)
    with torch.cuda.graph(qtm):
        c.Qtm(g, one, a, 0.16, 0.01)
    ref = O.Qtm(dims, U, psi, 0.16, 0.01)
    eager = c.Qtm(g, c.empty(vh, "f64"), a, 0.16, 0.01)   # makes the fixed-point scratch
    assert rel(c.unpack(eager, vh, "f64").cpu().numpy(), ref) < 1e-13
    for o in (*outs, one):
        o.zero_()
    qtm.replay()
    nd.replay()
    torch.cuda.synchronize()
    assert rel(c.unpack(one, vh, "f64").cpu().numpy(), ref) < 1e-13
    assert all(np.array_equal(c.unpack(o, vh, "f64").cpu().numpy(), w) for o, w in zip(outs, want))
    g.close()
    c.close()


@pytest.mark.parametrize("prec,tol", [("f32", 1e-6), ("f64", 1e-13)])   # FP32 with the staged hop's tables, FP64 without
def test_batch_in_a_capture(prec, tol):
    """A batch that is new to the context (here: of a known shape, on other buffers) is refused by a capturing
    stream and leaves the batch before it in place; one that is in place is captured and replays."""
    from paper_1311_4521_gb300 import tmhop
    dims, n = (8, 8, 8, 8), 3
    vh = int(np.prod(dims)) // 2
    U = F.gauge_field(dims, 951, "random")
    psi = [F.gaussian_spinor(vh, 951, k) for k in range(2 * n)]
    c = tmhop.Context(0)
    g = c.gauge(dims, U, prec, 12 if prec == "f32" else 18)
    ins = [c.pack(p, prec) for p in psi]
    outs = [c.empty(vh, prec).zero_() for _ in psi]
    want = [O.Qtm(dims, U, p, 0.16, 0.01) for p in psi]

    def ok(ks):
        return all(rel(c.unpack(outs[k], vh, prec).cpu().numpy(), want[k]) < tol for k in ks)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        c.Qtm_batch([g] * n, outs[:n], ins[:n], 0.16, 0.01)
        torch.cuda.synchronize()
        assert ok(range(n))
    refused, taken = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(refused, stream=side):
        with pytest.raises(tmhop.TmError):
            c.Qtm_batch([g] * n, outs[n:], ins[n:], 0.16, 0.01)
    with torch.cuda.graph(taken, stream=side):
        c.Qtm_batch([g] * n, outs[:n], ins[:n], 0.16, 0.01)
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    taken.replay()
    torch.cuda.synchronize()
    assert ok(range(n)) and not any(bool(o.any()) for o in outs[n:])
    with torch.cuda.stream(side):
        c.Qtm_batch([g] * n, outs[n:], ins[n:], 0.16, 0.01)
        torch.cuda.synchronize()
        assert ok(range(n, 2 * n))
        for k in range(40):   # more tables than the pinned memory holds, buffers changing from call to call
            o = outs[k % 2:] + outs[:k % 2]
            c.Qtm_batch([g] * n, o[:n], ins[:n], 0.16, 0.01 + k)
        c.Qtm_batch([g] * n, outs[:n], ins[:n], 0.16, 0.01)
        torch.cuda.synchronize()
        assert ok(range(n))
    g.close()
    c.close()


def test_first_qtm_while_another_stream_captures():
    """With the scratch of the other operators in place, a first FP64 Q_tm on a stream of its own leaves the capture
    of another operator on another stream alone."""
    from paper_1311_4521_gb300 import tmhop
    dims = (8, 8, 8, 8)
    vh = int(np.prod(dims)) // 2
    U, psi = F.gauge_field(dims, 952, "random"), F.gaussian_spinor(vh, 952, 1)
    c = tmhop.Context(0)
    g, lo = c.gauge(dims, U, "f64", 18), c.gauge(dims, U, "f32", 12)
    a, a32, out, out32 = c.pack(psi, "f64"), c.pack(psi, "f32"), c.empty(vh, "f64"), c.empty(vh, "f32")
    c.Qnd(g, [c.empty(vh, "f64"), c.empty(vh, "f64")], [a, a], 0.16, 0.01, 0.02)
    torch.cuda.synchronize()
    graph, own = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph):   # global mode
        c.Qtm(lo, out32, a32, 0.16, 0.01)
        tmhop.tm_Qtm(c.handle, g.handle, out, a, 0.16, 0.01, 1, own)
    torch.cuda.synchronize()
    out32.zero_()
    graph.replay()
    torch.cuda.synchronize()
    want = O.Qtm(dims, U, psi, 0.16, 0.01)
    assert rel(c.unpack(out, vh, "f64").cpu().numpy(), want) < 1e-13
    assert rel(c.unpack(out32, vh, "f32").cpu().numpy(), want) < 1e-6
    for h in (g, lo):
        h.close()
    c.close()
