"""What is measured: the calls that a program using this library makes.

Every case goes through the public entry points (``tmhop.Context`` and
``autograd``) on fields that such a program holds on the GPU: a gauge handle,
packed spinor fields, and for the differentiation and host cases the torch
tensors themselves.  One context serves the whole process, as in a program.

``exact`` restates the operators in plain torch on complex128 tensors over the
full lattice (``torch.roll`` for the neighbours), sharing nothing with the
library.
"""
from __future__ import annotations

import math

import torch

from paper_1311_4521_gb300 import autograd, tmhop

RECON = {"f64": (18, 12), "f64x": (18, 12), "f32": (12, 18), "f16": (12,)}
# kappa and mu of the two link ensembles: near-thermalised links exp(0.3 i A), and random SU(3)
PARAMS = {"near": (0.1394, 0.0015), "random": (0.16, 0.01)}
CG_TOL = 1e-12


# ------------------------------------------------------------------ cases
def _case(op, prec, recon, dims, **more):
    c = {"op": op, "prec": prec, "recon": recon, "lx": dims[0], "ly": dims[1], "lz": dims[2], "lt": dims[3],
         "links": "near"}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the operator on the plain small lattice with random links, where launches count
        dict(_case("qtm", "f64", 18, (8, 8, 8, 8), links="random", sign=1), name="qtm_f64_8x8x8x8"),
        # the production lattice in full precision: the library's headline workload
        dict(_case("qtm", "f64", 18, (32, 32, 32, 64), sign=1), name="qtm_f64_32x32x32x64"),
        # the operator inside a single-precision iteration, two-row links, an ensemble's medium lattice
        dict(_case("qtm", "f32", 12, (20, 20, 20, 40), sign=-1), name="qtm_f32_20x20x20x40"),
        # one adjoint hop in half precision storage, the inner format of the fastest mixed solver
        dict(_case("hop", "f16", 12, (28, 28, 28, 56), dir=0, dagger=True), name="hop_f16_28x28x28x56"),
        # one hop in double-float storage on a small lattice whose half-row is no power of two
        dict(_case("hop", "f64x", 18, (12, 12, 12, 24), dir=1, dagger=False), name="hop_f64x_12x12x12x24"),
        # twelve right-hand sides (one source per spin and colour) on the production lattice in one call
        dict(_case("batch", "f32", 12, (32, 32, 32, 64), nlat=1, nrhs=12), name="batch_f32_12rhs_32x32x32x64"),
        # an ensemble of small lattices in one call
        dict(_case("batch", "f32", 12, (8, 8, 8, 8), nlat=64, nrhs=1), name="batch_f32_64lat_8x8x8x8"),
        # an inversion: mixed-precision CG, FP32 inside, FP64 reliable updates
        dict(_case("cg", "f32", 12, (24, 24, 24, 48)), name="cg_f32_24x24x24x48"),
        # the fermion force of a molecular-dynamics step in full precision
        dict(_case("force", "f64", 18, (16, 16, 16, 32), mode=0), name="force_f64_16x16x16x32"),
        # backpropagation through the operator: forward and the gradients of spinor and links
        dict(_case("autograd", "f32", 12, (24, 24, 24, 32)), name="autograd_f32_24x24x24x32"),
        # the mass-split doublet
        dict(_case("nd", "f32", 12, (24, 24, 24, 48), sign=1), name="nd_f32_24x24x24x48"),
        # fields in host memory, copied in and out around the operator
        dict(_case("host", "f64", 18, (24, 24, 24, 48), nrhs=4), name="host_f64_24x24x24x48"),
    ]


def _even_dims(rng, lo, hi):
    """Four even extents, at least 4, whose volume is spread over [lo, hi] on a logarithmic scale."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = (want / 2) ** 0.25
    while True:
        d = [max(4, 2 * round(side * rng.uniform(0.75, 1.3) / 2)) for _ in range(3)]
        t = max(4, 2 * round(want / (d[0] * d[1] * d[2]) / 2))
        if 0.7 * lo <= d[0] * d[1] * d[2] * t <= hi:
            return (d[0], d[1], d[2], t)


def draw(rng):
    """One more case: an operator call more often than the composed ones, over all storage formats."""
    op = rng.choice(["qtm", "qtm", "qtm", "hop", "hop", "batch", "batch", "cg", "force", "autograd", "nd", "host"])
    vmax = {"qtm": 32 ** 3 * 64, "hop": 32 ** 3 * 64, "batch": 32 ** 3 * 64}.get(op, 24 ** 3 * 48)
    precs = {"batch": ["f64", "f32", "f32", "f16"], "cg": ["f64", "f32", "f32", "f16"], "force": ["f64", "f32"],
             "autograd": ["f64", "f32"], "nd": ["f64", "f32", "f16"], "host": ["f64", "f32"]}
    prec = rng.choice(precs.get(op, ["f64", "f64", "f64x", "f32", "f32", "f16"]))
    recons = RECON[prec]
    recon = recons[0] if op in ("batch", "autograd") or rng.random() < 0.7 else recons[-1]
    more = {}
    if op == "qtm":
        more = {"sign": rng.choice([1, -1])}
    elif op == "hop":
        more = {"dir": rng.choice([0, 1]), "dagger": rng.random() < 0.5}
    elif op == "batch":
        more = rng.choice([{"nlat": 1, "nrhs": rng.randint(2, 12)}, {"nlat": rng.randint(2, 64), "nrhs": 1}])
        vmax //= max(1, more["nlat"]) if more["nrhs"] == 1 else 4
    elif op == "force":
        more = {"mode": rng.choice([0, 1])}
    elif op == "nd":
        more = {"sign": rng.choice([1, -1])}
    elif op == "host":
        more = {"nrhs": rng.randint(1, 4)}
    c = _case(op, prec, recon, _even_dims(rng, 512, vmax), **more)
    if op in ("qtm", "hop") and rng.random() < 0.3:
        c["links"] = "random"
    return c


# ------------------------------------------------------------------ inputs
def _dims(case):
    return (case["lx"], case["ly"], case["lz"], case["lt"])


def _vh(case):
    return case["lx"] * case["ly"] * case["lz"] * case["lt"] // 2


def _unit_rows(a, b):
    """SU(3) matrices from two rows each: Gram-Schmidt, third row conj(row0 x row1)."""
    a = a / torch.linalg.vector_norm(a, dim=1, keepdim=True)
    b = b - (a.conj() * b).sum(1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b, dim=1).conj()], dim=1)


def _links(n, kind, gen):
    """n SU(3) matrices: random ones, or near the identity (1 + iA - A^2/2 with A = 0.3 sum w_a lambda_a / 2,
    w_a ~ N(0, 1), made unitary)."""
    dev = "cuda"
    if kind == "random":
        z = torch.randn((2, n, 3), dtype=torch.complex128, device=dev, generator=gen)
        return _unit_rows(z[0], z[1])
    w = 0.15 * torch.randn((8, n), dtype=torch.float64, device=dev, generator=gen)
    A = torch.zeros((n, 3, 3), dtype=torch.complex128, device=dev)
    s = 1 / math.sqrt(3.0)
    A[:, 0, 0], A[:, 1, 1], A[:, 2, 2] = w[2] + s * w[7], -w[2] + s * w[7], -2 * s * w[7]
    for (i, j), (p, q) in (((0, 1), (0, 1)), ((0, 2), (3, 4)), ((1, 2), (5, 6))):
        A[:, i, j] = torch.complex(w[p], -w[q])
        A[:, j, i] = torch.complex(w[p], w[q])
    rows = []
    for k in range(2):
        r = 1j * A[:, k] - 0.5 * sum(A[:, k, m, None] * A[:, m] for m in range(3))
        r[:, k] += 1
        rows.append(r)
    return _unit_rows(rows[0], rows[1])


def _inputs(case, seed):
    """Link fields (4, V, 3, 3) and spinor fields (V/2, 4, 3), complex128 on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    vh = _vh(case)
    U = [torch.stack([_links(2 * vh, case["links"], gen) for _ in range(4)]) for _ in range(case.get("nlat", 1))]
    count = {"batch": case.get("nlat", 1) * case.get("nrhs", 1), "nd": 2, "autograd": 2, "host": case.get("nrhs", 1)}
    psi = [torch.randn((vh, 4, 3), dtype=torch.complex128, device="cuda", generator=gen)
           for _ in range(count.get(case["op"], 1))]
    return U, psi


def prepare(case, seed):
    op, prec, recon, dims = case["op"], case["prec"], case["recon"], _dims(case)
    ctx = autograd.context(0)
    U, psi = _inputs(case, seed)
    s = {"case": case, "ctx": ctx, "vh": _vh(case)}
    if op == "autograd":
        s["U"], s["psi"], s["g"] = U[0].requires_grad_(True), psi[0].requires_grad_(True), psi[1]
        return s
    if op == "cg":
        s["hi"] = ctx.gauge(dims, U[0], "f64", 18)
        s["lo"] = None if prec == "f64" else ctx.gauge(dims, U[0], prec, recon)
        s["b"], s["x"] = ctx.pack(psi[0], "f64"), ctx.empty(s["vh"], "f64")
        return s
    gauges = [ctx.gauge(dims, u, prec, recon) for u in U]
    if op == "host":
        s["g"] = gauges[0]
        s["in"] = [p.cpu().pin_memory() for p in psi]
        s["out"] = [torch.empty_like(p).pin_memory() for p in s["in"]]
        return s
    s["g"] = gauges if op == "batch" else gauges[0]
    if op == "batch" and case["nlat"] == 1:
        s["g"] = gauges * case["nrhs"]
    s["in"] = [ctx.pack(p, prec) for p in psi]
    if op != "force":
        s["out"] = [ctx.empty(s["vh"], prec) for _ in psi]
    return s


# ------------------------------------------------------------------ one pass
def _values(s, buf, prec):
    """The numbers of a packed field: its stored components (and site norms), or the double-float pairs' sums."""
    if prec == "f64":
        return buf.view(torch.float64)
    if prec == "f32":
        return buf.view(torch.float32)
    if prec == "f16":
        return [buf[:48 * s["vh"]].view(torch.float16), buf[48 * s["vh"]:].view(torch.float32)]
    return s["ctx"].unpack(buf, s["vh"], prec)


def run(s):
    case, ctx = s["case"], s["ctx"]
    op, prec = case["op"], case["prec"]
    kappa, mu = PARAMS[case["links"]]
    if op == "qtm":
        ctx.Qtm(s["g"], s["out"][0], s["in"][0], kappa, mu, case["sign"])
    elif op == "hop":
        ctx.hopping_eo(s["g"], s["out"][0], s["in"][0], case["dir"], case["dagger"])
    elif op == "batch":
        ctx.Qtm_batch(s["g"], s["out"], s["in"], kappa, mu)
    elif op == "nd":
        ctx.Qnd(s["g"], s["out"], s["in"], kappa, mu, 0.0018, case["sign"])
    elif op == "host":
        return ctx.Qtm_host(s["g"], s["out"], s["in"], kappa, mu)
    elif op == "force":
        return ctx.force(s["g"], s["in"][0], kappa, mu, case["mode"])
    elif op == "cg":
        s["x"].zero_()
        ctx.cg(s["hi"], s["x"], s["b"], kappa, mu, CG_TOL, 30000, s["lo"])
        return _values(s, s["x"], "f64")
    elif op == "autograd":
        out = autograd.qtm(s["psi"], s["U"], _dims(case), kappa, mu, prec)
        gpsi, gU = torch.autograd.grad(out, (s["psi"], s["U"]), s["g"])
        return {"out": out.detach(), "grad_psi": gpsi, "grad_U": gU}
    return [_values(s, o, prec) for o in s["out"]]


# ------------------------------------------------------------------ work
SPINOR = {"f64": 192, "f64x": 192, "f32": 96, "f16": 52}
LINK = {("f64", 18): 144, ("f64", 12): 96, ("f64x", 18): 144, ("f64x", 12): 96, ("f32", 18): 72, ("f32", 12): 48,
        ("f16", 12): 24}
CANON_U, CANON_PSI = 144, 192   # canonical complex double: one link matrix, one spinor
HOP_FLOP, QTM_FLOP = 1320, 2 * 1320 + 168


def _qtm_bytes(prec, recon, n=1):
    """Q_tm per even site for n right-hand sides of one lattice: input read and output written once, links of both
    parities read once (8 per even-odd pair of sites); the odd temporary is written and read."""
    return n * 4 * SPINOR[prec] + 8 * LINK[prec, recon]


def work(case):
    op, prec, recon, vh = case["op"], case["prec"], case["recon"], _vh(case)
    f, l8 = SPINOR[prec], 8 * LINK[prec, recon]
    if op == "hop":
        return {"bytes": vh * (2 * f + l8), "flops": vh * HOP_FLOP}
    if op == "qtm":
        return {"bytes": vh * _qtm_bytes(prec, recon), "flops": vh * QTM_FLOP}
    if op == "batch":
        n = case["nlat"] * case["nrhs"]
        return {"bytes": vh * case["nlat"] * _qtm_bytes(prec, recon, case["nrhs"]), "flops": vh * n * QTM_FLOP}
    if op == "nd":
        return {"bytes": vh * (8 * f + l8), "flops": 2 * vh * (QTM_FLOP + 96)}
    if op == "host":   # in and out over the host link, and the operator
        n = case["nrhs"]
        return {"bytes": n * vh * (2 * CANON_PSI + _qtm_bytes(prec, recon)), "flops": n * vh * QTM_FLOP}
    if op == "force":  # X read, links of both parities read, the force field written; three hops and the outer products
        return {"bytes": vh * (f + l8 + 8 * CANON_U), "flops": vh * (3 * HOP_FLOP + 8 * 400)}
    if op == "cg":     # about 150 iterations of two Q_tm and the vector updates
        return {"bytes": 150 * vh * (2 * _qtm_bytes(prec, recon) + 6 * f), "flops": 150 * vh * (2 * QTM_FLOP + 200)}
    # autograd: links, psi and the upstream gradient read, output and both gradients written
    return {"bytes": vh * (2 * 8 * CANON_U + 4 * CANON_PSI), "flops": vh * (2 * QTM_FLOP + 2 * HOP_FLOP + 8 * 300)}


# ------------------------------------------------------------------ 64-bit values
def _gammas():
    z, o = torch.zeros((2, 2), dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
    pauli = [torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128),
             torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128),
             torch.tensor([[1, 0], [0, -1]], dtype=torch.complex128)]
    g = [torch.cat([torch.cat([z, -o], 1), torch.cat([-o, z], 1)], 0)]
    g += [torch.cat([torch.cat([z, -1j * p], 1), torch.cat([1j * p, z], 1)], 0) for p in pauli]
    return [m.cuda() for m in g]


class _Plain:
    """The operators in plain torch on the full lattice, complex128; antiperiodic in time, direction 0 is time."""

    AXIS = (0, 3, 2, 1)   # axis of direction mu in the (t, z, y, x) grid

    def __init__(self, dims, U):
        self.grid = tuple(reversed(dims))
        self.U = U
        t, z, y, x = torch.meshgrid(*[torch.arange(n, device="cuda") for n in self.grid], indexing="ij")
        par = ((t + z + y + x) & 1).reshape(-1)
        self.sites = [torch.nonzero(par == p).reshape(-1) for p in (0, 1)]
        self.gamma = _gammas()
        sign = torch.ones(self.grid, dtype=torch.float64, device="cuda")
        sign[-1] = -1
        self.last_t = sign.reshape(-1, 1, 1)
        self.g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda").reshape(4, 1)

    def _shift(self, f, mu, by):
        """f(x + mu) for by = -1, f(x - mu) for by = +1."""
        return torch.roll(f.reshape(self.grid + f.shape[1:]), by, self.AXIS[mu]).reshape(f.shape)

    @staticmethod
    def _mul(m, v):
        return sum(m[:, None, :, b] * v[:, :, b, None] for b in range(3))

    def _spin(self, mu, s, v):
        """(1 + s gamma_mu) v: each row of gamma_mu has one entry."""
        g = self.gamma[mu]
        col = g.abs().argmax(1).tolist()
        return v + s * torch.stack([g[a, col[a]] * v[:, col[a]] for a in range(4)], 1)

    def hop(self, psi, to, dagger=False):
        """The hop from the other parity to parity `to`; the adjoint swaps the projectors."""
        full = psi.new_zeros((self.last_t.shape[0], 4, 3)).index_copy(0, self.sites[1 - to], psi)
        s = 1 if dagger else -1
        out = 0
        for mu in range(4):
            sg = self.last_t if mu == 0 else 1.0
            fwd = self._mul(self.U[mu], self._shift(full, mu, -1))
            out = out + sg * self._spin(mu, s, fwd)
            bwd = self._mul(self.U[mu].mH, sg * full)
            out = out + self._spin(mu, -s, self._shift(bwd, mu, 1))
        return out[self.sites[to]]

    def qtm(self, psi, kappa, mu):
        w = 1j * 2 * kappa * mu * self.g5
        t = self.hop(psi, 1) / (1 + w)
        return self.g5 * ((1 + w) * psi - kappa ** 2 * self.hop(t, 0))

    def qnd(self, s, c, kappa, mu_sigma, mu_delta):
        mb, eb = 1j * 2 * kappa * mu_sigma * self.g5, 2 * kappa * mu_delta
        d = 1 - mb * mb - eb * eb

        def inv(a, b):
            return ((1 - mb) * a + eb * b) / d, ((1 + mb) * b + eb * a) / d

        ts, tc = inv(self.hop(s, 1), self.hop(c, 1))
        return (self.g5 * ((1 + mb) * s - eb * c - kappa ** 2 * self.hop(ts, 0)),
                self.g5 * ((1 - mb) * c - eb * s - kappa ** 2 * self.hop(tc, 0)))


def _solve(P, b, kappa, mu, tol=1e-14, maxiter=400):
    """CG on Q(-mu) Q(mu) x = b."""
    x, r = torch.zeros_like(b), b.clone()
    p, rr = r.clone(), torch.sum(r.abs() ** 2).item()
    stop = tol ** 2 * rr
    for _ in range(maxiter):
        if rr <= stop:
            break
        q = P.qtm(p, kappa, mu)
        alpha = rr / torch.sum(q.abs() ** 2).item()
        x += alpha * p
        r -= alpha * P.qtm(q, kappa, -mu)
        new = torch.sum(r.abs() ** 2).item()
        p = r + (new / rr) * p
        rr = new
    return x


def _stored(v, prec):
    """A spinor field (V/2, 4, 3) laid out as _values gives it."""
    vh, c = v.shape[0], torch.view_as_real(v.reshape(v.shape[0], 12).resolve_conj().contiguous())
    if prec == "f64":
        return c.permute(1, 0, 2).reshape(-1)
    if prec == "f32":
        return c.reshape(vh, 6, 4).permute(1, 0, 2).reshape(-1)
    if prec == "f16":
        norm = c.abs().amax((1, 2))
        return [(c / norm[:, None, None]).reshape(vh, 3, 8).permute(1, 0, 2).reshape(-1), norm]
    return v


def exact(case, seed):
    op, prec, dims = case["op"], case["prec"], _dims(case)
    kappa, mu = PARAMS[case["links"]]
    U, psi = _inputs(case, seed)
    P = _Plain(dims, U[0])
    if op == "qtm":
        return [_stored(P.qtm(psi[0], kappa, case["sign"] * mu), prec)]
    if op == "hop":
        return [_stored(P.hop(psi[0], case["dir"], case["dagger"]), prec)]
    if op == "batch":
        if case["nlat"] == 1:
            return [_stored(P.qtm(p, kappa, mu), prec) for p in psi]
        return [_stored(_Plain(dims, u).qtm(p, kappa, mu), prec) for u, p in zip(U, psi)]
    if op == "nd":
        return [_stored(o, prec) for o in P.qnd(psi[0], psi[1], kappa, case["sign"] * mu, 0.0018)]
    if op == "host":
        return [P.qtm(p, kappa, mu).cpu() for p in psi]
    if op == "cg":
        return _stored(_solve(P, psi[0], kappa, mu), "f64")
    if op == "autograd":
        P.U, x = U[0].requires_grad_(True), psi[0].requires_grad_(True)
        out = P.qtm(x, kappa, mu)
        gpsi, gU = torch.autograd.grad(out, (x, P.U), psi[1])
        return {"out": out.detach(), "grad_psi": gpsi, "grad_U": gU}
    # force: dS = -2 Re <Y, dQ X> with Y = Q X; F = -TA(U G^dag) / 2
    X = psi[0]
    with torch.no_grad():
        Y = P.qtm(X, kappa, mu)
    P.U = U[0].requires_grad_(True)
    (G,) = torch.autograd.grad(-2 * torch.sum((Y.conj() * P.qtm(X, kappa, mu)).real), P.U)
    if case["mode"] == 1:
        return G
    W = (U[0].detach().reshape(-1, 3, 3, 1) * G.conj().transpose(-1, -2).reshape(-1, 1, 3, 3)).sum(2).reshape(G.shape)
    A = 0.5 * (W - W.mH)
    tr = torch.diagonal(A, dim1=-2, dim2=-1).sum(-1) / 3
    return -0.5 * (A - tr[..., None, None] * torch.eye(3, dtype=A.dtype, device=A.device))
