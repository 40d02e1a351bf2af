"""Link buffers handed from destroyed gauge handles to new ones: results with
handles of changing sizes and formats, a handle replaced while launches of
another stream still read its links, handles that outlive their context, and
the memory given back."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu
TOL = {"f64": 1e-13, "f32": 1e-6, "f16": 5e-3}


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def test_reused_buffers_hold_the_new_links():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    for k, (dims, prec, recon) in enumerate([((8, 8, 8, 8), "f64", 18), ((8, 8, 8, 8), "f64", 12), ((8, 6, 8, 8), "f64", 18),
                                             ((8, 8, 8, 16), "f32", 18), ((8, 8, 8, 16), "f32", 12), ((8, 8, 8, 8), "f64", 18),
                                             ((8, 8, 8, 16), "f16", 12)]):
        vh = int(np.prod(dims)) // 2
        U, psi = F.gauge_field(dims, 930 + k, "random"), F.gaussian_spinor(vh, 930, k)
        g = c.gauge(dims, U, prec, recon)
        out = c.Qtm(g, c.empty(vh, prec), c.pack(psi, prec), 0.16, 0.01)
        g.close()   # with the launches still in flight
        assert rel(c.unpack(out, vh, prec).cpu().numpy(), O.Qtm(dims, U, psi, 0.16, 0.01)) < TOL[prec]
    c.close()


def test_links_read_on_another_stream_are_not_overwritten():
    from paper_1311_4521_gb300 import tmhop
    dims = (16, 16, 16, 16)
    vh = int(np.prod(dims)) // 2
    c = tmhop.Context(0)
    U0, U1 = (F.gauge_field(dims, s, "near", 0.3) for s in (940, 941))
    src = c.pack(F.gaussian_spinor(vh, 940, 1), "f32")
    g = c.gauge(dims, U0, "f32", 12)
    ref = c.hopping_eo(g, c.empty(vh, "f32"), src, 0).clone()
    outs = [c.empty(vh, "f32") for _ in range(200)]
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        for o in outs:
            c.hopping_eo(g, o, src, 0)
    g.close()
    g = c.gauge(dims, U1, "f32", 12)   # takes the buffer once the launches above are done
    torch.cuda.synchronize()
    assert all(torch.equal(o, ref) for o in outs)
    g.close()
    c.close()


def test_handles_may_outlive_their_context_and_memory_is_given_back():
    from paper_1311_4521_gb300 import tmhop
    dims = (16, 16, 16, 32)
    U = torch.zeros((4, 16 ** 3 * 32, 3, 3), dtype=torch.complex128)
    U[..., 0, 0] = U[..., 1, 1] = U[..., 2, 2] = 1
    U = U.cuda()
    c = tmhop.Context(0)
    c.gauge(dims, U, "f64", 18).close()
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]   # one spare buffer held
    g, h = c.gauge(dims, U, "f64", 18), c.gauge(dims, U, "f64", 18)
    c.close()
    g.close()
    h.close()
    assert torch.cuda.mem_get_info()[0] >= free0
