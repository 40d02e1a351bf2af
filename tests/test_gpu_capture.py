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
