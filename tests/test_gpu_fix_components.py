"""The fixed-point FP64 hop, component by component: the error of every real
and imaginary part against the sum of the absolute products that enter it,
which is what bounds the error of FP64 products and sums.  Links that do not
mix colours, and fields with components of very different size, some of them
zero, are where an error relative to a site's largest component would show."""
import numpy as np
import pytest

from paper_1311_4521_gb300 import fields as F
from test_gpu_fix import Extended, apply

pytestmark = pytest.mark.gpu
KAPPA, MU = 0.1394, 0.0015
# FP64: a projection, chains of 12 multiply-adds per direction, 8 sums: 20 roundings of at most 2^-53 S each, S the
# sum of the absolute products.  Fixed point: 0.35 2^-53 S rms where S is the smallest that is taken (1.3 the most in
# thousands of samples), and the conversion's rounding.
K = 20 * 2.0 ** -53
SMALL, LARGE = ((6, 4, 2, 10), (1, -1, -1, -1)), ((18, 10, 14, 12), (-1, 1, 1, 1))


@pytest.fixture(scope="module")
def ctx():
    from paper_1311_4521_gb300 import tmhop
    c = tmhop.Context(0)
    yield c
    c.close()


def gauge(dims, kind):
    if kind in ("random", "near"):
        return F.gauge_field(dims, 981, kind, 0.3)
    if kind == "smooth":
        return F.gauge_field(dims, 981, "near", 1e-6)
    V = int(np.prod(dims))
    rng = np.random.default_rng(981)
    U = np.zeros((4, V, 3, 3), dtype=np.complex128)
    if kind == "unit":
        U[...] = np.eye(3)
    elif kind == "diagonal":
        a = rng.uniform(-np.pi, np.pi, size=(2, 4, V))
        for k, phase in enumerate((a[0], a[1], -a[0] - a[1])):
            U[..., k, k] = np.exp(1j * phase)
    elif kind == "block":   # SU(2) on two colours
        q = rng.normal(size=(4, 4, V))
        q /= np.sqrt((q ** 2).sum(0))
        a, b = q[0] + 1j * q[1], q[2] + 1j * q[3]
        U[..., 0, 0], U[..., 0, 1], U[..., 1, 0], U[..., 1, 1] = a, b, -b.conj(), a.conj()
        U[..., 2, 2] = 1
    else:                   # "real": rotations
        m = rng.normal(size=(4, V, 3, 3))
        m[..., 0, :] /= np.linalg.norm(m[..., 0, :], axis=-1, keepdims=True)
        m[..., 1, :] -= (m[..., 1, :] * m[..., 0, :]).sum(-1, keepdims=True) * m[..., 0, :]
        m[..., 1, :] /= np.linalg.norm(m[..., 1, :], axis=-1, keepdims=True)
        m[..., 2, :] = np.cross(m[..., 0, :], m[..., 1, :])
        U[...] = m
    return U


def field(dims, kind):
    vh = int(np.prod(dims)) // 2
    rng = np.random.default_rng(982)
    psi = F.gaussian_spinor(vh, 982, 1)
    if kind == "graded":        # 24 parts of fixed sizes between 1 and 2^-45
        f = 2.0 ** -rng.permutation(np.linspace(0, 45, 24)).round().reshape(2, 4, 3)
        return psi.real * f[0] + 1j * psi.imag * f[1]
    if kind == "per_component":
        e = rng.integers(0, 40, size=(2,) + psi.shape)
        return psi.real * 2.0 ** -e[0] + 1j * psi.imag * 2.0 ** -e[1]
    if kind == "one_component":   # diluted in spin and colour
        psi[:, (0, 1, 3)] = 0
        psi[..., 1:] = 0
        return psi
    if kind == "real":
        return psi.real + 0j
    if kind == "wave":            # a plane wave: with unit links sums cancel to rounding
        k = np.arange(vh)
        return (np.exp(2j * np.pi * k / 7)[:, None, None] * np.ones((vh, 4, 3))).astype(np.complex128)
    if kind == "sites":
        return psi * 2.0 ** -rng.integers(0, 60, size=(vh, 1, 1))
    return psi


class Absolute(Extended):
    """Sums of absolute products; a complex number holds those of the real and of the imaginary part."""

    @staticmethod
    def mul(a, b):
        return (a.real * b.real + a.imag * b.imag) + 1j * (a.real * b.imag + a.imag * b.real)

    @staticmethod
    def mod(a):
        return np.abs(a.real) + 1j * np.abs(a.imag)

    def sums(self, psi, to, dagger=False, projected=True):
        """Of the hop of psi; projected=False: with |a| + |b| for the projections' a + b as well (psi's own errors)."""
        full = np.zeros((self.U.shape[1], 4, 3), dtype=np.clongdouble)
        full[self.sites[1 - to]] = psi
        s, out, sign, self.bc = (1 if dagger else -1), 0, self.bc, (1, 1, 1, 1)
        A = self.mod(self.U)
        for mu in range(4):
            for q, fwd in ((s, True), (-s, False)):
                P = np.eye(4) + q * self.gamma[mu]
                h = np.einsum("st,xta->xsa", P, full)
                if not projected:
                    h = sum(self.mul(np.broadcast_to(self.mod(P[:, t])[:, None], full.shape[1:]), full[:, t:t + 1])
                            for t in range(4))
                h = self.mod(h)
                if fwd:
                    g = self.shift(h, mu, -1)
                    out = out + sum(self.mul(A[mu][:, None, :, b], g[:, :, b:b + 1]) for b in range(3))
                else:
                    g = sum(self.mul(A[mu][:, None, b, :], h[:, :, b:b + 1]) for b in range(3))
                    out = out + self.shift(g, mu, 1)
        self.bc = sign
        return out[self.sites[to]]

    def qtm_bound(self, psi, kappa, mu):
        w = np.longdouble(2 * kappa * mu)
        twist = lambda v: v + w * (v.imag + 1j * v.real)   # |1 + i w g5| times v
        t = self.hop(psi, 1) / (1 + 1j * w * self.g5)
        first = twist(self.sums(psi, 1))
        return twist(self.mod(psi)) + np.longdouble(kappa) ** 2 * (self.sums(t, 0) + self.sums(first, 0, projected=False))


def within(got, want, size):
    err = Absolute.mod(got - want)
    return bool(np.all(err.real <= K * size.real) and np.all(err.imag <= K * size.imag))


CASES = [(SMALL, 18, links, kind) for links in ("random", "near", "smooth", "unit", "diagonal", "block", "real")
         for kind in ("gauss", "graded", "per_component", "one_component", "real", "wave", "sites")]
CASES += [(SMALL, 12, links, kind) for links in ("random", "unit", "diagonal") for kind in ("graded", "one_component", "sites")]
CASES += [(LARGE, 18, "near", "graded"), (LARGE, 18, "diagonal", "per_component"), (LARGE, 12, "unit", "graded"),
          (LARGE, 18, "random", "one_component"), (LARGE, 18, "block", "wave")]


@pytest.mark.parametrize("lattice,recon,links,kind", CASES)
def test_every_component(ctx, lattice, recon, links, kind):
    dims, bc = lattice
    U, psi = gauge(dims, links), field(dims, kind)
    if recon == 12:
        U[..., 2, :] = np.cross(U[..., 0, :], U[..., 1, :]).conj()
    E = Absolute(dims, U, bc)
    g = ctx.gauge(dims, U, "f64", recon, bc)
    for op in ((0, False), (1, True)) if lattice is SMALL else ((1, False),):
        assert within(apply(ctx, g, psi, op), E.hop(psi, *op), E.sums(psi, *op)), op
    want, bound = E.qtm(psi, KAPPA, MU), E.qtm_bound(psi, KAPPA, MU)
    got = apply(ctx, g, psi, "qtm", KAPPA, MU)
    assert within(got, want, bound)
    if recon == 18 and lattice is SMALL:   # FP64 products throughout meet the same bound
        assert within(apply(ctx, g, psi, "batch", KAPPA, MU), want, bound)
    g.close()


@pytest.mark.parametrize("lattice", [SMALL, LARGE])
@pytest.mark.parametrize("kind", ["gauss", "graded", "one_component"])
def test_host_fields_give_the_same_bits(ctx, lattice, kind):
    import torch
    dims, bc = lattice
    psi = field(dims, kind)
    g = ctx.gauge(dims, gauge(dims, "near"), "f64", 18, bc)
    a, o = torch.from_numpy(psi).pin_memory(), torch.empty(psi.shape, dtype=torch.complex128).pin_memory()
    ctx.Qtm_host(g, [o], [a], KAPPA, MU)
    assert np.array_equal(o.numpy(), apply(ctx, g, psi, "qtm", KAPPA, MU))
    g.close()


@pytest.mark.parametrize("lattice,recon", [(SMALL, 18), (SMALL, 12), (LARGE, 18)])
@pytest.mark.parametrize("links,keep", [("near", "spin"), ("near", "spin, real"), ("unit", "spin"), ("unit", "component"),
                                        ("diagonal", "component"), ("real", "colour, real")])
def test_exact_zeros_stay_with_the_integers(ctx, lattice, recon, links, keep):
    """Fields diluted in spin and colour: components that nothing but zeros enters do not send their sites to FP64
    products.  Those would give the bits of a handle without a fixed-point copy at every site; the integers round some
    sums the other way (unit links, real fields: few of the nonzero components' sums are rounded at all)."""
    from paper_1311_4521_gb300 import tmhop
    dims, bc = lattice
    U, psi = gauge(dims, links), field(dims, "gauss")
    if recon == 12:
        U[..., 2, :] = np.cross(U[..., 0, :], U[..., 1, :]).conj()
    if "real" in keep:
        psi = psi.real + 0j
    if "spin" in keep or "component" in keep:
        psi[:, (0, 1, 3)] = 0
    if "colour" in keep or "component" in keep:
        psi[..., (0, 2)] = 0
    E = Absolute(dims, U, bc)
    g = ctx.gauge(dims, U, "f64", recon, bc)
    tmhop.tm_ctx_set_fixed_point(ctx.handle, False)
    products = ctx.gauge(dims, U, "f64", recon, bc)
    tmhop.tm_ctx_set_fixed_point(ctx.handle, True)
    got = apply(ctx, g, psi, (1, False))
    assert within(got, E.hop(psi, 1, False), E.sums(psi, 1, False))
    assert not np.array_equal(got, apply(ctx, products, psi, (1, False)))
    if lattice is SMALL:
        assert within(apply(ctx, g, psi, "qtm", KAPPA, MU), E.qtm(psi, KAPPA, MU), E.qtm_bound(psi, KAPPA, MU))
    products.close()
    g.close()
