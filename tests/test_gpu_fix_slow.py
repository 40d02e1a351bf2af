"""Sites that the fixed-point FP64 hop leaves to FP64 products (tm_fix.cuh),
in CTAs that also hold threads past the lattice's end: the operator and the
solver's hops against references, over boundary signs in space and both link
formats."""
import numpy as np
import pytest

import oracle as O
from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu
KAPPA, MU = 0.1394, 0.0015
EPS = 2.0 ** -52
# 15120 and 15840 sites per parity: beyond the split hop, with a partial last CTA of 64
SIGNED = [((18, 10, 14, 12), (-1, 1, 1, 1), 18), ((22, 6, 10, 24), (1, -1, 1, -1), 12)]


@pytest.fixture(scope="module")
def ctx():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    yield c
    c.close()


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def wide(vh, seed):
    """A Gaussian field with components of every eighth site 2^-40 to 2^-30 of the others': their neighbours are
    slow sites, one to all of a warp's."""
    rng = np.random.default_rng(seed)
    psi = F.gaussian_spinor(vh, seed, 1)
    psi[::8] *= 2.0 ** -rng.integers(30, 41, size=psi[::8].shape)
    return psi


@pytest.mark.parametrize("dims,bc,recon", SIGNED)
def test_slow_sites_next_to_threads_past_the_end(ctx, dims, bc, recon):
    vh = int(np.prod(dims)) // 2
    U, psi = F.gauge_field(dims, 961, "near", 0.3), wide(vh, 961)
    g, src = ctx.gauge(dims, U, "f64", recon, bc), ctx.pack(psi, "f64")
    outs = [ctx.Qtm(g, ctx.empty(vh, "f64"), src, KAPPA, MU) for _ in range(20)]
    got = [ctx.unpack(o, vh, "f64").cpu().numpy() for o in outs]
    assert rel(got[0], O.Qtm(dims, U, psi, KAPPA, MU, bc=bc)) < 8 * EPS   # the operator's error and the oracle's, each below EPS or a few
    assert all(np.array_equal(got[0], v) for v in got)
    g.close()


@pytest.mark.parametrize("inner", ["f64", "f32"])
@pytest.mark.parametrize("dims,bc,recon", SIGNED)
def test_solve_with_a_source_of_wide_range(ctx, dims, bc, recon, inner):
    """A point source: the first iterations meet slow sites in every hop.  FP64 CG takes the oracle's iterations
    but for rounding; what a wrong hop or update costs is more of them, or a residual that does not follow."""
    vh = int(np.prod(dims)) // 2
    U = F.gauge_field(dims, 962, "near", 0.3)
    b = np.zeros((vh, 4, 3), dtype=np.complex128)
    b[vh // 3, 1, 2] = 1.0
    b[vh // 2] = 2.0 ** -35 * (1 - 0.5j)
    g = ctx.gauge(dims, U, "f64", recon, bc)
    lo = None if inner == "f64" else ctx.gauge(dims, U, inner, 12, bc)
    x = ctx.empty(vh, "f64").zero_()
    st, info = ctx.cg(g, x, ctx.pack(b, "f64"), 0.12, 0.05, 1e-10, 1000, lo)
    assert st == 0 and info["true_relres"] <= 1e-10
    xs = ctx.unpack(x, vh, "f64").cpu().numpy()
    back = O.Qtm(dims, U, O.Qtm(dims, U, xs, 0.12, 0.05, bc=bc), 0.12, -0.05, bc=bc)
    assert rel(back, b) < 2e-10
    if inner == "f64":
        iters = O.cg_QdagQ(dims, U, b, 0.12, 0.05, 1e-10, 1000, bc=bc)[1]
        assert abs(info["iters"] - iters) <= 1 + iters // 50
    g.close()
    if lo:
        lo.close()


@pytest.mark.parametrize("recon", [18, 12])
@pytest.mark.parametrize("which", ["one", "all"])
@pytest.mark.parametrize("scale", [1.3 * 2.0 ** -59, 1e-20, 1e-120, 0.0])
def test_tiny_links_are_not_taken_for_zero(ctx, recon, which, scale):
    """Links below the fixed-point unit act with what they are; links of exact zeros do nothing."""
    dims = (4, 4, 4, 4)
    V = 4 ** 4
    U, psi = F.gauge_field(dims, 963, "random"), F.gaussian_spinor(V // 2, 963, 1)
    rows = (slice(None), 7) if which == "one" else (slice(None), slice(None))
    U[rows] = 0.0 if scale == 0.0 else U[rows] * scale
    if recon == 12:
        U[..., 2, :] = np.cross(U[..., 0, :], U[..., 1, :]).conj()
    g, src = ctx.gauge(dims, U, "f64", recon), ctx.pack(psi, "f64")
    for to in (0, 1):
        got = ctx.unpack(ctx.hopping_eo(g, ctx.empty(V // 2, "f64"), src, to), V // 2, "f64").cpu().numpy()
        want = O.hopping(dims, U, psi, to)
        assert np.abs(got - want).max() <= 64 * EPS * np.abs(want).max()
        for mu in range(4) if which == "one" else ():   # what enters through the changed links alone
            only = np.zeros_like(U)
            only[mu, 7] = U[mu, 7]
            h = ctx.gauge(dims, only, "f64", recon)
            got = ctx.unpack(ctx.hopping_eo(h, ctx.empty(V // 2, "f64"), src, to), V // 2, "f64").cpu().numpy()
            want = O.hopping(dims, only, psi, to)
            assert np.abs(got - want).max() <= 64 * EPS * np.abs(want).max()
            assert bool(want.any()) == (scale != 0.0)
            h.close()
    g.close()
