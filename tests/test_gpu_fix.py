"""The FP64 hop with fixed-point link products: its error against extended
precision next to that of FP64 products, its fallback on sites it does not
take (wide ranges, extreme exponents, NaN, Inf), its edges (lattices with
partial blocks of 32 and 64 sites, boundary signs in every direction, tiled
maps) and the gauge fields that get no fixed-point links.

tm_Qtm_batch multiplies with FP64 products and serves as the other path."""
import numpy as np
import pytest

from paper_1311_4521_gb300 import fields as F

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def ctx():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    yield c
    c.close()


class Extended:
    """The operators in numpy long double on the full lattice."""

    def __init__(self, dims, U, bc):
        self.grid, self.bc, self.U = tuple(reversed(dims)), bc, U.astype(np.clongdouble)
        idx = np.indices(self.grid).sum(0).reshape(-1) & 1
        self.sites = [np.flatnonzero(idx == p) for p in (0, 1)]
        s = [np.array([[0, 1], [1, 0]]), np.array([[0, -1j], [1j, 0]]), np.array([[1, 0], [0, -1]])]
        z, o = np.zeros((2, 2)), np.eye(2)
        self.gamma = [np.block([[z, -o], [-o, z]])] + [np.block([[z, -1j * p], [1j * p, z]]) for p in s]
        self.g5 = np.array([1, 1, -1, -1], dtype=np.longdouble)[:, None]

    def shift(self, f, mu, by):
        """f(x + mu) for by = -1, f(x - mu) for by = 1, with the boundary sign of the hop."""
        ax = (0, 3, 2, 1)[mu]
        v = np.roll(f.reshape(self.grid + f.shape[1:]), by, ax)
        edge = [slice(None)] * v.ndim
        edge[ax] = -1 if by < 0 else 0
        v[tuple(edge)] *= self.bc[mu]
        return v.reshape(f.shape)

    def hop(self, psi, to, dagger=False):
        full = np.zeros((self.U.shape[1], 4, 3), dtype=np.clongdouble)
        full[self.sites[1 - to]] = psi
        s, out = (1 if dagger else -1), 0
        for mu in range(4):
            P = [np.eye(4) + q * self.gamma[mu] for q in (s, -s)]
            fwd = np.einsum("xab,xsb->xsa", self.U[mu], self.shift(full, mu, -1))
            bwd = self.shift(np.einsum("xba,xsb->xsa", self.U[mu].conj(), full), mu, 1)
            out = out + np.einsum("st,xta->xsa", P[0], fwd) + np.einsum("st,xta->xsa", P[1], bwd)
        return out[self.sites[to]]

    def qtm(self, psi, kappa, mu):
        w = 1j * np.longdouble(2 * kappa * mu) * self.g5
        return self.g5 * ((1 + w) * psi - np.longdouble(kappa) ** 2 * self.hop(self.hop(psi, 1) / (1 + w), 0))

    def neighbour_sum(self, a, to):
        """Sum over the 8 neighbours of a per-site number of the other parity."""
        full = np.zeros(self.U.shape[1])
        full[self.sites[1 - to]] = a
        v = full.reshape(self.grid)
        return sum(np.roll(v, by, ax) for ax in range(4) for by in (1, -1)).reshape(-1)[self.sites[to]]


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def apply(ctx, g, psi, op, kappa=0.1394, mu=0.0015):
    vh = psi.shape[0]
    src, out = ctx.pack(psi, "f64"), ctx.empty(vh, "f64")
    out.fill_(0xFF)
    if op == "qtm":
        ctx.Qtm(g, out, src, kappa, mu)
    elif op == "batch":
        ctx.Qtm_batch([g], [out], [src], kappa, mu)
    else:
        ctx.hopping_eo(g, out, src, *op)
    return ctx.unpack(out, vh, "f64").cpu().numpy()


def has_fixed_links(g):
    return g.nbytes > 8 * g.vh * g.reconstruct * 8


SMALL = [((4, 4, 4, 4), (-1, 1, 1, 1)), ((6, 4, 2, 10), (1, -1, -1, -1)), ((10, 6, 2, 2), (-1, -1, 1, 1))]
# beyond the lattices whose hops are split over warps, ragged; with and without boundary signs in space
LARGE = [((18, 10, 14, 12), (-1, 1, 1, 1), 18, "near"), ((14, 10, 18, 14), (1, 1, -1, 1), 12, "random")]


@pytest.mark.parametrize("dims,bc,recon,kind",
                         [(d, bc, r, k) for d, bc in SMALL for r in (18, 12) for k in ("random", "near")] + LARGE)
def test_error_is_no_larger_than_with_fp64_products(ctx, dims, bc, recon, kind):
    U = F.gauge_field(dims, 911, kind)
    psi = F.gaussian_spinor(int(np.prod(dims)) // 2, 911, 1)
    E = Extended(dims, U, bc)
    g = ctx.gauge(dims, U, "f64", recon, bc)
    assert has_fixed_links(g)
    want = E.qtm(psi, 0.1394, 0.0015)
    err = rel(apply(ctx, g, psi, "qtm"), want)
    assert err < EPS
    if recon == 18:   # the batched operator takes no 12-real FP64 links
        assert err <= 1.02 * rel(apply(ctx, g, psi, "batch"), want)
    for op in ((0, False), (1, False), (0, True), (1, True)):
        # conversions to FP64, the projections' rounding: below one unit of the last place in the norm
        assert rel(apply(ctx, g, psi, op), E.hop(psi, *op)) < EPS
    g.close()


RANGES = ["1e200", "1e-200", "1e-290", "per_site", "per_component", "zero_sites", "point", "all_zero"]
RANGE_CASES = [(r, (4, 6, 4, 8), k) for r in (18, 12) for k in RANGES] + [
    (18, (18, 10, 14, 12), k) for k in ("1e-290", "per_component", "zero_sites")]


def ranged(psi, kind):
    rng = np.random.default_rng(5)
    psi = psi.copy()
    if kind.startswith("1e"):
        return psi * float(kind)
    if kind == "per_site":
        return psi * 10.0 ** rng.integers(-12, 12, size=(len(psi), 1, 1))
    if kind == "per_component":
        return psi * 2.0 ** -rng.integers(0, 60, size=psi.shape)
    if kind == "zero_sites":
        psi[rng.random(len(psi)) < 0.7] = 0
        return psi
    if kind == "point":
        psi[...] = 0
        psi[len(psi) // 2, 1, 2] = 1
        return psi
    return psi * 0


@pytest.mark.parametrize("recon,dims,kind", RANGE_CASES)
def test_ranges(ctx, recon, dims, kind):
    """Every output component against extended precision, relative to the largest input components that enter it:
    8 roundings of the sums of 8 hops of magnitude at most 4 each."""
    bc = (-1, 1, 1, 1)
    U = F.gauge_field(dims, 912, "random")
    psi = ranged(F.gaussian_spinor(int(np.prod(dims)) // 2, 912, 1), kind)
    E = Extended(dims, U, bc)
    g = ctx.gauge(dims, U, "f64", recon, bc)
    big = np.abs(psi).max((1, 2))
    near = E.neighbour_sum(big, 0)
    tiny = 2.0 ** -1070
    assert np.all(np.abs(apply(ctx, g, psi, (0, False)) - E.hop(psi, 0)).max((1, 2)) <= 16 * EPS * near + tiny)
    bound = big + 0.1394 ** 2 * 4 * E.neighbour_sum(E.neighbour_sum(big, 1), 0)
    got = apply(ctx, g, psi, "qtm")
    assert np.all(np.abs(got - E.qtm(psi, 0.1394, 0.0015)).max((1, 2)) <= 16 * EPS * bound + tiny)
    if kind == "all_zero":
        assert np.all(got == 0)
    g.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e305])
@pytest.mark.parametrize("dims", [(8, 4, 4, 8), (18, 10, 14, 12)])
def test_values_that_are_not_finite_spread_as_with_fp64_products(ctx, bad, dims):
    U = F.gauge_field(dims, 913, "random")
    psi = F.gaussian_spinor(int(np.prod(dims)) // 2, 913, 1)
    psi[17, 2, 1] = bad
    g = ctx.gauge(dims, U, "f64", 18)
    a, b = apply(ctx, g, psi, "qtm").view(np.float64), apply(ctx, g, psi, "batch").view(np.float64)
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
    fine = np.isfinite(b)
    assert np.array_equal(a[~fine & ~np.isnan(b)], b[~fine & ~np.isnan(b)])
    small = fine & (np.abs(b) < 1e3)
    assert small.any() and np.abs(a[small] - b[small]).max() < 64 * EPS
    g.close()


@pytest.mark.parametrize("change", ["large", "nan", "weak", "wide_row"])
def test_links_far_from_su3_use_fp64_products(ctx, change):
    dims = (4, 4, 4, 4)
    U = F.gauge_field(dims, 914, "random")
    V = U.shape[1]
    if change == "large":
        U[2, V // 3, 1, 1] = 3.0
    elif change == "weak":
        U[1, 5] *= 1e-3
    elif change == "wide_row":
        U[0, 7, 2] = 0.7 + 0.7j
    g = ctx.gauge(dims, U, "f64", 18)
    assert not has_fixed_links(g) if change != "nan" else True
    psi = F.gaussian_spinor(V // 2, 914, 1)
    E = Extended(dims, U, (-1, 1, 1, 1))
    assert rel(apply(ctx, g, psi, "qtm"), E.qtm(psi, 0.1394, 0.0015)) < 4 * EPS
    g.close()
    if change == "nan":
        U[3, 3, 0, 0] = np.nan
        g = ctx.gauge(dims, U, "f64", 18)
        assert not has_fixed_links(g)
        assert np.isnan(apply(ctx, g, psi, (1, False)).view(np.float64)).any()
        g.close()


@pytest.mark.parametrize("dims,names", [((16, 4, 4, 6), ["linear32", "linear96", "box8x2x2x1", "box8x4x4x1"]),
                                        ((16, 8, 16, 16), ["linear32", "linear96", "box8x2x2x1", "box4x4x4x2"])])
def test_maps_give_identical_bits(ctx, dims, names):
    from paper_1311_4521_gb300 import tmhop
    U = F.gauge_field(dims, 915, "near", 0.3)
    psi = F.gaussian_spinor(int(np.prod(dims)) // 2, 915, 1)
    g = ctx.gauge(dims, U, "f64", 18)
    ref, hop = apply(ctx, g, psi, "qtm"), apply(ctx, g, psi, (1, True))
    for name in names:
        tmhop.tm_gauge_set_map(ctx.handle, g.handle, name)
        assert np.array_equal(apply(ctx, g, psi, "qtm"), ref), name
        assert np.array_equal(apply(ctx, g, psi, (1, True)), hop), name
    g.close()
