"""The work that users of this library have it do, as cases that can be timed and checked.

Every case goes through the public binding (paper_1303_1377_gb300.ddamg.Solver) on torch CUDA
tensors: the operator applications of a program with its own outer iteration (Dslash, smoother,
transfers, coarse operator, level-1 smoother), the part of the setup that rebuilds the
interpolation, and whole solves.  Gauge fields are exp(i eps H) with eps = 0.5 as in the
repository's workloads, drawn on the device from the seed; right-hand sides are complex Gaussian;
test vectors are Gaussian fields smoothed by a few Richardson steps, as those of an adaptive setup.

The V-cycle pieces of SINGLE and HALF handles compute in FP32 and return their FP32 numbers in
complex128 arrays (the ABI's only field type); the program here keeps them as complex64 Krylov
vectors, so run() returns them as that.
"""
from __future__ import annotations

import math

import torch

from paper_1303_1377_gb300 import ddamg

EPS, C_SW = 0.5, 1.0
M0 = -0.9  # the serving stream's lightest common mass: leftmost eigenvalue of D(0) about 0.99, so |eig| >= 0.09
PREC = {"double": ddamg.PREC_DOUBLE, "single": ddamg.PREC_SINGLE, "half": ddamg.PREC_HALF}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _case(kind, dims, nrhs, prec, name=None, block=(4, 4, 4, 4), n_vec=20, entry=""):
    c = {"kind": kind, "nrhs": nrhs, "prec": prec, "n_vec": n_vec, "entry": entry}
    for m in range(4):
        c["L%d" % m], c["b%d" % m] = dims[m], block[m]
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the smallest call: D on one FP32 field of a small lattice, as in a Lanczos or inverter step of
        # a single propagator component (launches and latency count)
        _case("dirac", (16, 16, 16, 16), 1, "single", "dslash_f32_16x16x16x16_1", entry="f32"),
        # D on the twelve spin-colour components of a propagator, larger than L2
        _case("dirac", (32, 32, 32, 32), 12, "half", "dslash_f32_32x32x32x32_12", entry="f32"),
        # the FP64-accurate product of FP32 fields that certifies residuals of the refinement
        _case("dirac", (24, 24, 24, 24), 12, "single", "dslash_mixed_24x24x24x24_12", entry="mixed"),
        # the smoother (two SAP iterations) of the half-precision V-cycle on a propagator batch:
        # the bulk of every solve of the headline configuration
        _case("smoother", (32, 32, 32, 32), 12, "half", "sap_half_32x32x32x32_12"),
        # the smoother of the default FP32 V-cycle on a single right-hand side
        _case("smoother", (16, 16, 16, 16), 1, "single", "sap_single_16x16x16x16_1"),
        # ragged: unequal extents and a partly filled batch, as a serving stream sends
        _case("smoother", (24, 8, 16, 40), 7, "half", "sap_half_24x8x16x40_7"),
        # restriction of a residual batch and prolongation of a coarse correction batch
        _case("transfer", (32, 32, 32, 32), 12, "half", "transfer_half_32x32x32x32_12"),
        # the coarse operator of the two-level solves of the serving stream
        _case("coarse", (32, 32, 32, 32), 12, "half", "coarse_half_32x32x32x32_12"),
        # the smoother of the second level in three-level solves
        _case("smoother1", (32, 32, 32, 32), 12, "half", "sap1_half_32x32x32x32_12"),
        # rebuilding the interpolation and the coarse operator from twenty test vectors: every round of
        # a setup, and every operator whose vectors are kept on disk
        _case("setup", (16, 16, 16, 16), 4, "single", "setup_single_16x16x16x16_20"),
        # whole solves: one right-hand side, two levels, FP32 V-cycle (the defaults) ...
        _case("solve", (16, 16, 16, 16), 1, "single", "solve_single_16x16x16x16_1"),
        # ... and a propagator batch, three levels, half-precision V-cycle
        _case("solve3", (32, 16, 16, 16), 12, "half", "solve3_half_32x16x16x16_12"),
    ]


def draw(rng):
    kind = rng.choice(["dirac", "dirac", "smoother", "smoother", "smoother", "transfer", "transfer", "coarse", "smoother1", "setup",
                       "solve", "solve3"])
    small = kind in ("setup", "solve", "solve3")
    step = 16 if kind in ("smoother1", "solve3") else 8
    top = 65536 if kind in ("setup", "solve") else 131072 if kind == "solve3" else 24**4 if kind != "smoother1" else 32**4
    want = math.exp(rng.uniform(math.log(step**4), math.log(top)))
    dims = [step] * 4
    while True:
        grown = [m for m in range(4) if dims[m] + step <= 48 and math.prod(dims) // dims[m] * (dims[m] + step) <= want]
        if not grown:
            break
        dims[rng.choice(grown)] += step
    if kind in ("smoother1", "solve3"):  # two even levels of blocks: extents that are multiples of 16
        dims = [d // 16 * 16 for d in dims]
    nrhs = rng.randint(1, 4) if kind == "setup" else rng.randint(1, 12)
    prec = rng.choice(["single", "half", "half"]) if not small or kind == "solve3" else "single"
    if kind == "setup":
        prec = rng.choice(["single", "half", "double"])
    if kind == "solve":
        nrhs = rng.randint(1, 4)
        prec = rng.choice(["single", "half"])
    entry = rng.choice(["f32", "f32", "f64", "mixed"]) if kind == "dirac" else ""
    if entry == "f64":
        prec = "double"
    block = (4, 4, 4, 4)
    if kind in ("dirac", "smoother", "transfer", "coarse") and rng.random() < 0.25:
        block = rng.choice([(2, 4, 4, 4), (4, 4, 2, 4), (4, 2, 2, 4)])
    n_vec = rng.choice([8, 12, 16, 20, 20, 24])
    return _case(kind, dims, nrhs, prec, block=block, n_vec=n_vec, entry=entry)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _dims(c):
    return tuple(c["L%d" % m] for m in range(4))


def _block(c):
    return tuple(c["b%d" % m] for m in range(4))


def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _gauss(shape, seed, stream, dtype=torch.complex128):
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=_gen(seed, stream), device="cuda", dtype=real))


def _mm(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(dims, seed):
    """U_mu(x) = exp(i eps H), H traceless hermitian Gaussian: [V, 4, 3, 3] complex128."""
    a = _gauss((math.prod(dims) * 4, 3, 3), seed, 1)
    h = 0.5 * (a + a.mH)
    eye = torch.eye(3, dtype=h.dtype, device="cuda")
    h = h - (h.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3)[:, None, None] * eye
    x = (0.25j * EPS) * h
    u = eye + x / 16
    for k in range(15, 0, -1):  # Taylor series of exp(x) at a quarter of the angle, squared twice
        u = eye + _mm(x, u) / k
    u = _mm(u, u)
    return _mm(u, u).reshape(math.prod(dims), 4, 3, 3).contiguous()


def _test_vectors(c, U, seed):
    """n_vec smoothed Gaussian fields [N, V, 4, 3]: three Richardson steps v <- v - D v / 5."""
    dims = _dims(c)
    op = _Wilson(dims, U.to(torch.complex64), M0, site=False)
    v = _gauss((c["n_vec"], math.prod(dims), 4, 3), seed, 2, torch.complex64).reshape((c["n_vec"],) + dims + (4, 3))
    for _ in range(3):
        v = v - 0.2 * op.apply(v)
    return v.reshape(c["n_vec"], math.prod(dims), 4, 3).to(torch.complex128).contiguous()


def _coarse_shape(c):
    nb = [c["L%d" % m] // c["b%d" % m] for m in range(4)]
    return math.prod(nb), 2 * c["n_vec"]


def _rhs(c, seed):
    dtype = torch.complex64 if c["entry"] in ("f32", "mixed") else torch.complex128
    return _gauss((c["nrhs"], math.prod(_dims(c)), 4, 3), seed, 3, dtype)


def _coarse_rhs(c, seed):
    return _gauss((c["nrhs"],) + _coarse_shape(c), seed, 4)


def prepare(case, seed):
    c, kind = case, case["kind"]
    dims = _dims(c)
    U = _links(dims, seed)
    p = ddamg.default_params(n_vec=c["n_vec"], block=_block(c), precision=PREC[c["prec"]], seed=int(seed) + 1, n_inv=2)
    if kind in ("solve", "solve3"):
        p.tol = 1e-12  # heavy-quark propagators fall by many orders of magnitude over the lattice
    torch.cuda.synchronize()
    s = ddamg.Solver(dims, U, M0, C_SW, p, setup=False)
    st = {"case": c, "s": s}
    if kind in ("dirac", "smoother", "transfer", "solve", "solve3", "setup"):
        st["x"] = _rhs(c, seed)
    if kind in ("transfer", "coarse", "smoother1", "setup"):
        st["e"] = _coarse_rhs(c, seed)
    if kind in ("transfer", "coarse", "smoother1"):
        s.setup_from_vectors(_test_vectors(c, U, seed))
    if kind == "setup":
        st["v"] = _test_vectors(c, U, seed)
    if kind in ("solve", "solve3"):
        s.run_setup()
    if kind == "smoother1":
        s.ml_build(_gauss((20,) + _coarse_shape(c), seed, 5), ddamg.ml_default_params(inner=1))
    if kind == "solve3":
        s.ml_setup(_gauss((20,) + _coarse_shape(c), seed, 5), ddamg.ml_default_params(inner=1, n_inv1=2))
    return st


def run(state):
    c, s = state["case"], state["s"]
    kind = c["kind"]
    low = (lambda t: t) if c["prec"] == "double" else (lambda t: t.to(torch.complex64))
    if kind == "dirac":
        return {"f32": s.apply_D_f32, "f64": s.apply_D, "mixed": s.apply_D_mixed}[c["entry"]](state["x"])
    if kind == "smoother":
        return low(s.apply_sap(state["x"], 2))
    if kind == "transfer":
        return [low(s.restrict(state["x"])), low(s.prolong(state["e"]))]
    if kind == "coarse":
        return low(s.apply_Dc(state["e"]))
    if kind == "smoother1":
        return low(s.ml_apply_sap1(state["e"], 2))
    if kind == "setup":  # the new interpolation and coarse operator, and their first use
        s.setup_from_vectors(state["v"])
        return [low(s.restrict(state["x"])), low(s.apply_Dc(state["e"]))]
    return (s.solve_zero_guess if kind == "solve" else s.ml_solve_zero_guess)(state["x"])[0]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
HOP, SITE = 168, 504  # flops of one hop (projection, two SU(3) products, reconstruction) and of one site term


def _sap_flops(V, h_in, hop, site, comps, mr, nu):
    """Flops of nu red-black SAP iterations: per pair of an even and an odd site the residual, the
    reduced right-hand side, mr minimal-residual steps and the back-substitution."""
    pair = 2 * (8 * hop + site) + site + h_in * hop + mr * (2 * h_in * hop + 2 * site + 12 * comps) + h_in * hop + site
    return nu * V / 2 * pair


def work(case):
    c, kind = case, case["kind"]
    V, nr, N = math.prod(_dims(c)), c["nrhs"], c["n_vec"]
    NB, nc = _coarse_shape(c)
    real = {"double": 8, "single": 4, "half": 2}[c["prec"]]  # stored size of the V-cycle's operators
    h_in = sum(2 * (b - 1) / b for b in _block(c))
    if kind == "dirac":
        i, o, m = {"f32": (8, 8, 4), "f64": (16, 16, 8), "mixed": (8, 16, 8)}[c["entry"]]
        return {"bytes": V * (144 * m + 12 * nr * (i + o)), "flops": V * nr * (8 * HOP + SITE)}
    fine, coarse = 12 * V * nr * 16, NB * nc * nr * 16
    if kind == "smoother":  # links, site terms and their even-site inverses once; b in, z out
        return {"bytes": V * 180 * real + 2 * fine, "flops": nr * _sap_flops(V, h_in, HOP, SITE, 12, 4, 2)}
    if kind == "transfer":  # P once per direction
        return {"bytes": 2 * (V * 12 * N * 2 * real + fine + coarse), "flops": 2 * nr * V * 12 * N * 8}
    op = NB * 9 * nc * nc * 2 * real
    if kind == "coarse":
        return {"bytes": op + 2 * coarse, "flops": nr * NB * 9 * nc * nc * 8}
    if kind == "smoother1":  # 2^4 blocks of level-1 sites
        return {"bytes": op + op / 18 + 2 * coarse, "flops": nr * _sap_flops(NB, 4, 8 * nc * nc, 8 * nc * nc, nc, 4, 2)}
    # orthonormalisation of the vectors, D on the 2N columns of P, and the products with P^H over the
    # block (self) and its eight faces
    if kind == "setup":
        faces = sum(2 / b for b in _block(c))
        build = V * 12 * N * N * 8 + V * 2 * N * (8 * HOP + SITE) / 2 + V * 12 * N * N * 8 * (1 + faces)
        return {"bytes": V * 12 * N * 16 * 2 + V * 144 * 8 + NB * 9 * nc * nc * 16 + fine + 2 * coarse, "flops": build}
    # solves: about 20 outer iterations, each one D, two SAP iterations and the transfers; the coarse
    # solves are not counted
    it = V * (8 * HOP + SITE) + _sap_flops(V, h_in, HOP, SITE, 12, 4, 2) + 2 * V * 12 * N * 8
    return {"bytes": 2 * fine + 20 * V * (12 * N * 4 * real + 180 * real + 576), "flops": 20 * nr * it}


# ---------------------------------------------------------------------------
# the same results in 64 bits, from the formulas of the method in plain torch
# ---------------------------------------------------------------------------
# gamma_mu = [[0, B_mu], [B_mu^H, 0]] in the chiral basis; B_mu has one entry per row: (column, factor)
_B = [[(1, 1j), (0, 1j)], [(1, -1), (0, 1)], [(0, 1j), (1, -1j)], [(0, 1), (1, 1)]]


def _B_apply(mu, x, dag):
    rows = [None, None]
    for i, (j, f) in enumerate(_B[mu]):
        if dag:
            rows[j] = complex(f).conjugate() * x[..., i, :]
        else:
            rows[i] = f * x[..., j, :]
    return torch.stack(rows, dim=-2)


def _su3(U, h):
    """U h for links U [*L, 3, 3] and half spinors h [r, *L, 2, 3]."""
    out = 0
    for b in range(3):
        out = out + U[..., None, :, b] * h[..., b, None]
    return out


class _Wilson:
    """The clover-improved Wilson operator on fields [r, L0, L1, L2, L3, 4, 3]."""

    def __init__(self, dims, U, m0, site=True):
        self.dims, self.m0 = dims, m0
        self.U = [U.reshape(dims + (4, 3, 3))[..., mu, :, :] for mu in range(4)]
        self.A = self._site_term() if site else None

    def _site_term(self):
        U = self.U
        gam = []
        for mu in range(4):
            g = torch.zeros(4, 4, dtype=torch.complex128)
            for i, (j, f) in enumerate(_B[mu]):
                g[i, 2 + j] = f
                g[2 + j, i] = complex(f).conjugate()
            gam.append(g)

        def at(m, *steps):
            f = U[m]
            for d, s in steps:
                f = torch.roll(f, -s, d)
            return f

        A = torch.zeros(self.dims + (2, 6, 6), dtype=torch.complex128, device="cuda")
        A += (self.m0 + 4) * torch.eye(6, dtype=A.dtype, device="cuda")
        for a in range(4):
            for b in range(a + 1, 4):
                q = _mm(_mm(at(a), at(b, (a, 1))), _mm(at(a, (b, 1)).mH, at(b).mH))
                q = q + _mm(_mm(at(b), at(a, (a, -1), (b, 1)).mH), _mm(at(b, (a, -1)).mH, at(a, (a, -1))))
                q = q + _mm(_mm(at(a, (a, -1)).mH, at(b, (a, -1), (b, -1)).mH), _mm(at(a, (a, -1), (b, -1)), at(b, (b, -1))))
                q = q + _mm(_mm(at(b, (b, -1)).mH, at(a, (b, -1))), _mm(at(b, (b, -1), (a, 1)), at(a).mH))
                F = q - q.mH
                gg = gam[a] @ gam[b]
                for h in range(2):
                    for s in range(2):
                        for t in range(2):
                            f = complex(gg[2 * h + s, 2 * h + t])
                            if f != 0:
                                A[..., h, 3 * s:3 * s + 3, 3 * t:3 * t + 3] -= (C_SW / 16 * f) * F
        return A

    def hop(self, psi, mu, sign, U=None):
        """-1/2 (I -+ gamma_mu) (x) U psi(x +- mu)."""
        U = self.U[mu] if U is None else U
        if sign > 0:
            psi = torch.roll(psi, -1, 1 + mu)
        h = psi[..., :2, :] - sign * _B_apply(mu, psi[..., 2:, :], False)
        g = _su3(U if sign > 0 else U.mH, h)
        out = -0.5 * torch.cat([g, -sign * _B_apply(mu, g, True)], dim=-2)
        return out if sign > 0 else torch.roll(out, 1, 1 + mu)

    def hops(self, psi, U=None):
        out = 0
        for mu in range(4):
            for sign in (1, -1):
                out = out + self.hop(psi, mu, sign, None if U is None else U[mu])
        return out

    def site(self, psi, A):
        x = psi.reshape(psi.shape[:-2] + (2, 6))
        y = 0
        for b in range(6):
            y = y + A[..., b] * x[..., b, None]
        return y.reshape(psi.shape)

    def apply(self, psi):
        d = (4 + self.m0) * psi if self.A is None else self.site(psi, self.A)
        return d + self.hops(psi)


def _coord(dims, mu):
    shape = [1] * 4
    shape[mu] = dims[mu]
    return torch.arange(dims[mu], device="cuda").reshape(shape)


class _FineLevel:
    """D split for SAP on blocks: fields [r, *L, 4, 3]."""

    def __init__(self, D, block):
        self.D, self.dims, self.block = D, D.dims, block
        # links that stay inside a block
        self.Uin = [D.U[mu] * ((_coord(D.dims, mu) + 1) % block[mu] != 0)[..., None, None] for mu in range(4)]
        self.Ainv = torch.linalg.inv(D.A)

    def apply(self, x):
        return self.D.apply(x)

    def inner(self, x):
        return self.D.hops(x, self.Uin)

    def diag(self, x):
        return self.D.site(x, self.D.A)

    def diag_inv(self, x):
        return self.D.site(x, self.Ainv)


class _CoarseLevel:
    """D_c as a nine-point stencil B[d][site] (d = 0 self, 1 + 2 mu for +mu, 2 + 2 mu for -mu): fields [r, *n, nc]."""

    def __init__(self, dims, B, block):
        self.dims, self.block, self.B = dims, block, B
        self.B0inv = torch.linalg.inv(B[0])

    def _mul(self, B, x):
        r = x.shape[0]
        y = torch.matmul(B, x.reshape(r, -1, x.shape[-1]).permute(1, 2, 0))
        return y.permute(2, 0, 1).reshape(x.shape)

    def _hops(self, x, inside):
        out = 0
        for mu in range(4):
            for sign in (1, -1):
                y = self._mul(self.B[1 + 2 * mu + (sign < 0)], torch.roll(x, -sign, 1 + mu))
                if inside:
                    at = _coord(self.dims, mu) + (1 if sign > 0 else 0)
                    y = y * (at % self.block[mu] != 0)[..., None]
                out = out + y
        return out

    def apply(self, x):
        return self.diag(x) + self._hops(x, False)

    def inner(self, x):
        return self._hops(x, True)

    def diag(self, x):
        return self._mul(self.B[0], x)

    def diag_inv(self, x):
        return self._mul(self.B0inv, x)


def _sap(op, b, nu, mr=4):
    """nu red-black SAP iterations on D z = b from z = 0, each block solved by mr odd-even minimal-residual steps."""
    dims, block, tail = op.dims, op.block, b.dim() - 5
    even = sum(_coord(dims, m) for m in range(4)) % 2 == 0
    red = sum(_coord(dims, m) // block[m] for m in range(4)) % 2 == 0
    one = (...,) + (None,) * tail

    def per_block(f):  # sum over components and over each block, spread back over its sites
        f = f.sum(dim=tuple(range(5, 5 + tail))) if tail else f
        shape = [f.shape[0]]
        for m in range(4):
            shape += [dims[m] // block[m], block[m]]
        s = f.reshape(shape).sum(dim=(2, 4, 6, 8), keepdim=True)
        return s.expand(shape).reshape(f.shape)[one]

    z = torch.zeros_like(b)
    for _ in range(nu):
        for colour in (red, ~red):
            E, O = (colour & even)[one], (colour & ~even)[one]
            r = b - op.apply(z)
            re = r * E
            rho = r * O - op.inner(op.diag_inv(re)) * O
            x = torch.zeros_like(r)
            for _ in range(mr):
                t = (op.diag(rho) - op.inner(op.diag_inv(op.inner(rho) * E))) * O
                den = per_block((t.conj() * t).real)
                al = per_block(t.conj() * rho) / torch.where(den > 0, den, torch.ones_like(den))
                x, rho = x + al * rho, rho - al * t
            z = z + x + op.diag_inv(re - op.inner(x) * E)
    return z


class _Aggregates:
    """P of the aggregates (block, chirality half) from test vectors: orthonormal bases Q [NB, 2, 6 Vb, N]."""

    def __init__(self, dims, block, v=None):
        self.dims, self.block = dims, block
        self.n = tuple(dims[m] // block[m] for m in range(4))
        if v is not None:
            q = self.gather(v)
            for _ in range(2):  # Cholesky QR, twice
                c = torch.linalg.cholesky(q.mH @ q, upper=True)
                q = torch.linalg.solve_triangular(c, q, upper=True, left=False)
            self.Q = q

    def gather(self, x):  # [r, *L, 4, 3] -> [NB, 2, 6 Vb, r]
        n, b, r = self.n, self.block, x.shape[0]
        x = x.reshape(r, n[0], b[0], n[1], b[1], n[2], b[2], n[3], b[3], 2, 6).permute(1, 3, 5, 7, 9, 2, 4, 6, 8, 10, 0)
        return x.reshape(math.prod(n), 2, 6 * math.prod(b), r)

    def scatter(self, y):
        n, b, r = self.n, self.block, y.shape[-1]
        y = y.reshape(n + (2,) + tuple(b) + (6, r)).permute(10, 0, 5, 1, 6, 2, 7, 3, 8, 4, 9)
        return y.reshape((r,) + tuple(self.dims) + (4, 3))

    def restrict(self, x):  # -> [r, NB, 2N]
        c = self.Q.mH @ self.gather(x)
        return c.permute(3, 0, 1, 2).reshape(x.shape[0], c.shape[0], -1)

    def prolong(self, e):
        r, nb, nc = e.shape
        return self.scatter(self.Q @ e.reshape(r, nb, 2, nc // 2).permute(1, 2, 3, 0))


def _coarse_stencil(D, agg, fine):
    """B_d = P^H (the part of D in direction d) P, as [9][NB, 2N, 2N]."""
    nb, _, rows, N = agg.Q.shape
    B = torch.zeros(9, nb, 2 * N, 2 * N, dtype=torch.complex128, device="cuda")
    for h in range(2):
        q = torch.zeros_like(agg.Q)
        q[:, h] = agg.Q[:, h]
        for j in range(0, N, 4):
            cols = agg.scatter(q[..., j:j + 4])
            at = slice(h * N + j, h * N + min(j + 4, N))
            B[0, :, :, at] = agg.restrict(D.site(cols, D.A) + fine.inner(cols)).permute(1, 2, 0)
            for mu in range(4):
                out = D.U[mu] - fine.Uin[mu]
                for sign in (1, -1):
                    B[1 + 2 * mu + (sign < 0), :, :, at] = agg.restrict(D.hop(cols, mu, sign, out)).permute(1, 2, 0)
    return B


def _solve(D, b, tol):
    """D^{-1} b by conjugate gradients on D^H D (D^H = Gamma5 D Gamma5), repeated on the true residual."""
    def dag(x):
        y = D.apply(torch.cat([x[..., :2, :], -x[..., 2:, :]], dim=-2))
        return torch.cat([y[..., :2, :], -y[..., 2:, :]], dim=-2)

    def dot(x, y):
        return (x.conj() * y).real.sum(dim=tuple(range(1, x.dim())), keepdim=True)

    z = torch.zeros_like(b)
    bn = dot(b, b).sqrt()
    for _ in range(4):
        r = b - D.apply(z)
        if float((dot(r, r).sqrt() / bn).max()) < tol:
            break
        x, s = torch.zeros_like(b), dag(r)
        p, g, g0 = s, dot(s, s), dot(s, s)
        for k in range(2000):
            q = D.apply(p)
            a = g / dot(q, q).clamp_min(1e-300)
            x = x + a * p
            r = r - a * q
            s = dag(r)
            g1 = dot(s, s)
            p = s + (g1 / g.clamp_min(1e-300)) * p
            g = g1
            if k % 25 == 24 and float((g / g0).max()) < 1e-18:
                break
        z = z + x
    return z


def exact(case, seed):
    c, kind, dims = case, case["kind"], _dims(case)
    U = _links(dims, seed)
    D = _Wilson(dims, U, M0)
    shape = (c["nrhs"],) + dims + (4, 3)
    flat = (c["nrhs"], math.prod(dims), 4, 3)
    if kind == "dirac":
        return D.apply(_rhs(c, seed).to(torch.complex128).reshape(shape)).reshape(flat)
    if kind == "smoother":
        return _sap(_FineLevel(D, _block(c)), _rhs(c, seed).reshape(shape), 2).reshape(flat)
    if kind in ("solve", "solve3"):
        return _solve(D, _rhs(c, seed).reshape(shape), 1e-14).reshape(flat)
    v = _test_vectors(c, U, seed).reshape((c["n_vec"],) + dims + (4, 3))
    agg = _Aggregates(dims, _block(c), v)
    del v
    if kind == "transfer":
        return [agg.restrict(_rhs(c, seed).reshape(shape)), agg.prolong(_coarse_rhs(c, seed)).reshape(flat)]
    e = _coarse_rhs(c, seed)
    if kind == "smoother1":
        B = _coarse_stencil(D, agg, _FineLevel(D, _block(c)))
        op = _CoarseLevel(agg.n, B, (2, 2, 2, 2))
        return _sap(op, e.reshape((c["nrhs"],) + agg.n + (-1,)), 2).reshape(e.shape)
    ec = agg.restrict(D.apply(agg.prolong(e)))
    return ec if kind == "coarse" else [agg.restrict(_rhs(c, seed).reshape(shape)), ec]
