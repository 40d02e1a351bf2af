"""The double-float hop split over four warps: lattices below and above the
size that takes it, partial blocks of 32 sites, boundary signs, adjoint and
both link storages, against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bc", [((2, 2, 2, 2), (-1, 1, 1, 1)), ((6, 4, 2, 10), (1, -1, -1, -1)),
                                     ((16, 16, 16, 8), (-1, 1, 1, 1)), ((22, 14, 18, 6), (-1, -1, 1, 1)),
                                     ((34, 30, 18, 18), (-1, 1, 1, 1))])
@pytest.mark.parametrize("recon", [18, 12])
def test_double_float_hops_match_oracle(dims, bc, recon):
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    vh = int(np.prod(dims)) // 2
    U, psi = F.gauge_field(dims, 950, "near", 0.3), F.gaussian_spinor(vh, 950, 1)
    g, src = c.gauge(dims, U, "f64x", recon, bc), c.pack(psi, "f64x")

    def rel(buf, want):
        got = c.unpack(buf, vh, "f64x").cpu().numpy()
        return np.linalg.norm(got - want) / np.linalg.norm(want)

    out = c.empty(vh, "f64x")
    for par, dag in ((0, False), (1, True)):
        out.fill_(0xFF)
        assert rel(c.hopping_eo(g, out, src, par, dag), O.hopping(dims, U, psi, par, dagger=dag, bc=bc)) < 1e-13
    out.fill_(0xFF)
    assert rel(c.Qtm(g, out, src, 0.1394, 0.0015, -1), O.Qtm(dims, U, psi, 0.1394, -0.0015, bc=bc)) < 1e-13
    g.close()
    c.close()
