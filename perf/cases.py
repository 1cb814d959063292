"""The work that users of the library have it do, as cases to be timed.

A case is one call (or one fixed sequence of calls) of the public entry
points on inputs drawn from a seed: the Dirac operator, the projection onto
the block basis, the coarse operator, the set-up of basis and coarse
operator, the estimator contraction and whole solves.  Lattices, blockings,
numbers of basis vectors, couplings and solver tolerances are those of the
repository's benchmark and test configurations.

Inputs are made with torch on the GPU: SU(3) links exp(i eps H) with Gaussian
H, Gaussian test vectors, Z2 or Gaussian sources.  ``exact`` evaluates the
definitions (complex128, torch only) on the same inputs.
"""
from __future__ import annotations

import math

import torch

import paper_2412_06347_gb300 as m

PREC = {"fp64": m.MGLMA_FP64, "fp32": m.MGLMA_FP32, "bf16": m.MGLMA_BF16, "fp16": m.MGLMA_FP16}
OPS = {"D": m.MGLMA_OP_D, "Ddag": m.MGLMA_OP_DDAG, "Q": m.MGLMA_OP_Q, "DdagD": m.MGLMA_OP_DDAGD}

# (eps, kappa, csw) of the repository's ensembles by their lattice scale
SMALL = (0.3, 0.12, 1.0)       # 8^4
MEDIUM = (0.2, 0.125, 1.7)     # 32x16^3
LARGE = (0.15, 0.1266, 1.9)    # 64x32^3
COUPLINGS = {"small": SMALL, "medium": MEDIUM, "large": LARGE}


def _case(name, what, L, nrhs, couplings, **more):
    return dict({"name": name, "what": what, "L0": L[0], "L1": L[1], "L2": L[2], "L3": L[3], "nrhs": nrhs,
                 "couplings": couplings}, **more)


def listed():
    return [
        # one spinor on the smallest lattice: a residual check inside an
        # analysis script; launches and latency count
        _case("dirac_fp64_8c_1", "dirac", (8, 8, 8, 8), 1, "small", op="D", prec="fp64"),
        # the twelve spin-colour columns of one point source, Hermitian operator
        _case("dirac_fp64_32x16c_12", "dirac", (32, 16, 16, 16), 12, "medium", op="Q", prec="fp64"),
        # a ragged group of seven in single precision, as a relaxation or a
        # Chebyshev filter of D^dag D applies it
        _case("dirac_fp32_48x24c_7", "dirac", (48, 24, 24, 24), 7, "medium", op="DdagD", prec="fp32"),
        # the largest single-precision application: one 16-source group
        _case("dirac_fp32_64x32c_16", "dirac", (64, 32, 32, 32), 16, "large", op="D", prec="fp32"),
        # low-mode projection T0 R0 psi of one point source's columns in FP64
        _case("project_fp64_32x16c_12", "project", (32, 16, 16, 16), 12, "medium", block=4, nv=16, prec="fp64",
              store="fp32"),
        # the same for a 16-source noise group at the benchmark's basis, on
        # the tensor cores
        _case("project_bf16_64x32c_16", "project", (64, 32, 32, 32), 16, "large", block=4, nv=24, prec="bf16",
              store="fp16"),
        # the coarse Hermitian operator of the benchmark for one group
        _case("coarse_64x32c_16", "coarse", (64, 32, 32, 32), 16, "large", block=4, nv=24, op="Q", prec="fp32"),
        # set-up of a new configuration: relaxed basis, coarse operator, export
        _case("setup_32x16c", "setup", (32, 16, 16, 16), 1, "medium", block=4, nv=16, n_smooth=5),
        # the correlator contraction of twelve noise sources
        _case("contract_48x24c_12", "contract", (48, 24, 24, 24), 12, "medium"),
        # whole solves: one source on the smallest lattice,
        _case("solve_8c_1", "solve", (8, 8, 8, 8), 1, "small", block=2, nv=8, pieces=False),
        # the twelve columns of a point source with the low-mode piece,
        _case("solve_pieces_32x16c_12", "solve", (32, 16, 16, 16), 12, "medium", block=4, nv=16, pieces=True),
        # and a 16-source group at the benchmark's set-up
        _case("solve_64x32c_16", "solve", (64, 32, 32, 32), 16, "large", block=4, nv=24, pieces=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: lattices from 8^4 to 64x32^3 (odd extents for the
    operators that need no blocking), 1 to 16 right-hand sides."""
    what = rng.choice(["dirac", "dirac", "dirac", "project", "project", "coarse", "contract", "setup", "solve", "solve"])
    nrhs = _log_int(rng, 1, 16)
    if what in ("dirac", "contract"):
        scale = math.exp(rng.uniform(math.log(6), math.log(26)))
        L = [max(4, int(round(scale * rng.uniform(0.8, 1.25)))) for _ in range(4)]
        L[0] = min(2 * L[0], 64)
        c = {"what": what, "couplings": rng.choice(["small", "medium", "large"])}
        if what == "dirac":
            c["op"] = rng.choice(["D", "D", "Ddag", "Q", "DdagD"])
            c["prec"] = rng.choice(["fp32", "fp64"])
    else:
        blocks = [_log_int(rng, 2, 6) for _ in range(4)]
        if what in ("setup", "solve"):
            blocks = [min(v, 4) for v in blocks]
        L = [4 * v for v in blocks]
        L[0] *= rng.choice([1, 2])
        c = {"what": what, "couplings": "medium", "block": 4, "nv": rng.choice([8, 16, 24])}
        if what == "project":
            c["prec"] = rng.choice(["fp64", "fp32", "bf16"])
            c["store"] = rng.choice(["fp32", "fp16"])
        elif what == "coarse":
            c["op"] = rng.choice(["D", "Ddag", "Q"])
            c["prec"] = rng.choice(["fp32", "fp32", "fp64"])
        elif what == "setup":
            c["n_smooth"] = rng.choice([3, 5])
            nrhs = 1
        else:
            c["pieces"] = rng.choice([False, False, True])
    c.update({"L0": L[0], "L1": L[1], "L2": L[2], "L3": L[3], "nrhs": nrhs})
    return c


# ------------------------------------------------------------------ inputs
def _L(case):
    return (case["L0"], case["L1"], case["L2"], case["L3"])


def _volume(case):
    return math.prod(_L(case))


def _gen(seed, part):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + part)
    return g


def _complex_randn(shape, gen):
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), generator=gen, device="cuda", dtype=torch.float64))


def _links(case, seed):
    """U = exp(i eps sum_a h_a lambda_a / 2) per site and direction, [V, 4, 3, 3].

    H is traceless and Hermitian, so H^3 = (tr H^2 / 2) H + det H and the
    exponential series is a quadratic in H with scalar coefficients."""
    eps = COUPLINGS[case["couplings"]][0]
    n = _volume(case) * 4
    h = torch.randn((8, n), generator=_gen(seed, 1), device="cuda", dtype=torch.float64) * (0.5 * eps)
    H = torch.zeros((n, 3, 3), device="cuda", dtype=torch.complex128)
    for (i, j), a in (((0, 1), 0), ((0, 2), 3), ((1, 2), 5)):
        H[:, i, j] = torch.complex(h[a], -h[a + 1])
        H[:, j, i] = torch.complex(h[a], h[a + 1])
    d8 = h[7] / math.sqrt(3.0)
    H[:, 0, 0] = (h[2] + d8).to(torch.complex128)
    H[:, 1, 1] = (d8 - h[2]).to(torch.complex128)
    H[:, 2, 2] = (-2.0 * d8).to(torch.complex128)
    H2 = torch.stack([torch.stack([sum(H[:, i, k] * H[:, k, j] for k in range(3)) for j in range(3)], -1)
                      for i in range(3)], -2)
    half_tr = 0.5 * (H2[:, 0, 0] + H2[:, 1, 1] + H2[:, 2, 2]).real
    det = (H[:, 0, 0] * (H[:, 1, 1] * H[:, 2, 2] - H[:, 1, 2] * H[:, 2, 1])
           - H[:, 0, 1] * (H[:, 1, 0] * H[:, 2, 2] - H[:, 1, 2] * H[:, 2, 0])
           + H[:, 0, 2] * (H[:, 1, 0] * H[:, 2, 1] - H[:, 1, 1] * H[:, 2, 0])).real
    p = [torch.ones_like(det), torch.zeros_like(det), torch.zeros_like(det)]  # H^k = p0 + p1 H + p2 H^2
    f = [torch.ones_like(det).to(torch.complex128), torch.zeros_like(H[:, 0, 0]), torch.zeros_like(H[:, 0, 0])]
    c = 1.0 + 0.0j
    for k in range(1, 26):
        p = [p[2] * det, p[0] + p[2] * half_tr, p[1]]
        c = c * 1j / k
        f = [f[q] + c * p[q] for q in range(3)]
    U = f[1][:, None, None] * H + f[2][:, None, None] * H2
    for i in range(3):
        U[:, i, i] += f[0]
    return U.reshape(-1, 4, 3, 3).contiguous()


def _spinors(case, seed, n, part=2, z2=False):
    shape = (n, _volume(case), 4, 3)
    if z2:
        r = torch.randint(0, 2, shape, generator=_gen(seed, part), device="cuda", dtype=torch.int8)
        return (2 * r - 1).to(torch.complex128)
    return _complex_randn(shape, _gen(seed, part))


def _coarse_volume(case):
    return _volume(case) // case["block"] ** 4


_context = None


def _ctx():
    """The one context a program keeps."""
    global _context
    if _context is None:
        _context = m.Context(0)
    return _context


class State:
    """Buffers and handles of one program; handles are freed with it."""

    def __init__(self):
        self.gauge = self.sub = self.coarse = None

    def __del__(self):
        torch.cuda.synchronize()
        if self.coarse:
            m.mglma_coarse_free(self.coarse)
        if self.sub:
            m.mglma_subspace_free(self.sub)
        if self.gauge:
            m.mglma_gauge_free(self.gauge)


def prepare(case, seed):
    s, what, n, L = State(), case["what"], case["nrhs"], _L(case)
    s.case, s.ctx = case, _ctx()
    blk = (case.get("block", 4),) * 4
    V = _volume(case)
    if what == "contract":
        s.a = _spinors(case, seed, 3 * n, 2)
        s.b = _spinors(case, seed, n, 3)
        s.out = torch.zeros((n, L[0]), device="cuda", dtype=torch.complex128)
        torch.cuda.synchronize()
        return s
    eps, kappa, csw = COUPLINGS[case["couplings"]]
    U = _links(case, seed)
    torch.cuda.synchronize()
    s.gauge = m.mglma_gauge_load(s.ctx, L, U, kappa, csw)
    del U
    if what in ("project", "coarse"):
        # Gaussian test vectors: after the block orthonormalisation the basis
        # has the scale of any other, and the kernels do not see the rest
        vecs = _spinors(case, seed, case["nv"], 4)
        torch.cuda.synchronize()
        s.sub = m.mglma_subspace_load(s.ctx, s.gauge, blk, case["nv"], vecs, PREC[case.get("store", "fp32")])
        del vecs
    if what == "solve":
        # the benchmark's recipe: 5 MR steps, then 60 CG steps in FP32
        s.sub = m.mglma_subspace_create(s.ctx, s.gauge, blk, case["nv"], 5, int(seed), m.MGLMA_FP16, n_cg=60,
                                        cg_prec=m.MGLMA_FP32)
    if what in ("coarse", "solve"):
        s.coarse = m.mglma_coarse_build(s.ctx, s.gauge, s.sub, m.MGLMA_BF16)
    if what == "dirac":
        s.b = _spinors(case, seed, n)
        s.x = torch.zeros_like(s.b)
    elif what == "project":
        s.b = _spinors(case, seed, n)
        s.c = torch.zeros((n, _coarse_volume(case), 2 * case["nv"]), device="cuda", dtype=torch.complex128)
        s.x = torch.zeros_like(s.b)
    elif what == "coarse":
        s.b = _complex_randn((n, _coarse_volume(case), 2 * case["nv"]), _gen(seed, 2))
        s.x = torch.zeros_like(s.b)
    elif what == "setup":
        nv2 = 2 * case["nv"]
        s.x = torch.zeros((9, _coarse_volume(case), nv2, nv2), device="cuda", dtype=torch.complex128)
        s.seed = int(seed)
    elif what == "solve":
        # relative residual 1e-12, as the repository's tests of the pieces and
        # the estimator ask for, so that solutions agree to FP64 purposes
        s.prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, tol=1e-12)
        s.b = _spinors(case, seed, n, z2=True)
        s.x = torch.zeros_like(s.b)
        s.x1 = torch.zeros_like(s.b) if case["pieces"] else None
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return s


def run(s):
    case, what, n = s.case, s.case["what"], s.case["nrhs"]
    if what == "dirac":
        m.mglma_dirac_apply(s.ctx, s.gauge, OPS[case["op"]], n, s.b, s.x, PREC[case["prec"]])
        return s.x
    if what == "project":
        m.mglma_restrict(s.ctx, s.sub, n, s.b, s.c, PREC[case["prec"]])
        m.mglma_prolong(s.ctx, s.sub, n, s.c, s.x, PREC[case["prec"]])
        return {"coarse": s.c, "fine": s.x}
    if what == "coarse":
        m.mglma_coarse_apply(s.ctx, s.coarse, n, s.b, s.x, PREC[case["prec"]], op=OPS[case["op"]])
        return s.x
    if what == "setup":
        sub = m.mglma_subspace_build(s.ctx, s.gauge, (case["block"],) * 4, case["nv"], case["n_smooth"], s.seed,
                                     m.MGLMA_FP16)
        c = m.mglma_coarse_build(s.ctx, s.gauge, sub, m.MGLMA_BF16)
        m.mglma_coarse_export(c, s.x)
        m.mglma_coarse_free(c)
        m.mglma_subspace_free(sub)
        return s.x
    if what == "contract":
        m.mglma_contract(s.ctx, _L(case), n, s.a, s.b, s.out)
        return s.out
    m.mglma_solve_batch(s.ctx, s.gauge, s.coarse, s.prm, [n], s.b, s.x, s.x1)
    return {"x": s.x, "x_coarse": s.x1} if case["pieces"] else {"x": s.x}


def work(case):
    """Inputs read once, outputs written once, and the arithmetic of the
    definition (a solve: that of ten applications of D, one per decimal digit
    of the benchmark's residual)."""
    V, n, what = _volume(case), case["nrhs"], case["what"]
    spinors = 192.0 * V * n
    if what == "dirac":
        k = 2 if case["op"] == "DdagD" else 1
        fixed = 1152.0 * V if case["prec"] == "fp64" else 480.0 * V
        return {"bytes": fixed + 2 * spinors, "flops": 1896.0 * k * V * n}
    if what == "contract":
        return {"bytes": 4 * spinors, "flops": 288.0 * V * n}
    nv = case["nv"]
    V1 = _coarse_volume(case)
    if what == "project":
        basis = 2 * nv * 6 * V * {"fp64": 16.0, "fp32": 8.0, "bf16": 4.0}[case["prec"]]
        return {"bytes": basis + 2 * spinors + 2 * 16.0 * n * V1 * 2 * nv, "flops": 2 * 8.0 * 12 * nv * V * n}
    if what == "coarse":
        size = 16.0 if case["prec"] == "fp64" else 4.0
        return {"bytes": size * 9 * V1 * (2 * nv) ** 2 + 2 * 16.0 * n * V1 * 2 * nv,
                "flops": 8.0 * 9 * V1 * (2 * nv) ** 2 * n}
    if what == "setup":
        return {"bytes": 1152.0 * V + 16.0 * 9 * V1 * (2 * nv) ** 2,
                "flops": nv * (case["n_smooth"] + 2) * 1896.0 * V + 9 * 8.0 * (2 * nv) ** 2 * 6 * V}
    return {"bytes": 480.0 * V + 2 * nv * 6 * 4.0 * V + 4.0 * 9 * V1 * (2 * nv) ** 2
            + (3 if case["pieces"] else 2) * spinors, "flops": 10 * 1896.0 * V * n}


# ------------------------------------------------------------------ 64-bit definitions
def _gammas():
    s = [torch.tensor(v, dtype=torch.complex128) for v in
         ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
    e = [-torch.eye(2, dtype=torch.complex128)] + [-1j * v for v in s]
    out = []
    for k in range(4):
        g = torch.zeros((4, 4), dtype=torch.complex128)
        g[:2, 2:] = e[k]
        g[2:, :2] = e[k].conj().T
        out.append(g.cuda())
    return out


class _Dirac:
    """D = A - 1/2 sum_mu [(1 - g_mu) U_mu(x) T_mu + (1 + g_mu) T_mu^dag U_mu(x)^dag]
    on [n, V, 4, 3], antiperiodic in x0, A the clover term with the mass."""

    def __init__(self, case, seed):
        _, kappa, csw = COUPLINGS[case["couplings"]]
        self.L = _L(case)
        self.U = _links(case, seed).reshape(self.L + (4, 3, 3))
        self.U = [self.U[..., mu, :, :].contiguous() for mu in range(4)]
        self.g = _gammas()
        self.diag = 0.5 / kappa  # 4 + m0
        self.F = []
        for mu in range(4):
            for nu in range(mu + 1, 4):
                sigma = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                # sum over both orders of (mu, nu): twice the i/4 of the action
                self.F.append((0.5j * csw * sigma, self._field(mu, nu)))

    @staticmethod
    def _mul(*f):
        r = f[0]
        for q in f[1:]:
            r = torch.matmul(r, q)
        return r

    def _field(self, mu, nu):
        def at(f, *steps):  # f(x + steps)
            for d, k in steps:
                f = torch.roll(f, -k, d)
            return f

        def dag(f):
            return f.conj().transpose(-1, -2)
        Um, Un = self.U[mu], self.U[nu]
        Q = self._mul(Um, at(Un, (mu, 1)), dag(at(Um, (nu, 1))), dag(Un))
        Q = Q + self._mul(Un, dag(at(Um, (mu, -1), (nu, 1))), dag(at(Un, (mu, -1))), at(Um, (mu, -1)))
        Q = Q + self._mul(dag(at(Um, (mu, -1))), dag(at(Un, (mu, -1), (nu, -1))), at(Um, (mu, -1), (nu, -1)),
                          at(Un, (nu, -1)))
        Q = Q + self._mul(dag(at(Un, (nu, -1))), at(Um, (nu, -1)), at(Un, (mu, 1), (nu, -1)), dag(Um))
        return (Q - dag(Q)) / 8.0

    @staticmethod
    def _colour(M, v):  # [..., 3, 3] on [..., 4, 3]
        return torch.matmul(v, M.transpose(-1, -2))

    @staticmethod
    def _spin(G, v):  # [4, 4] on [..., 4, 3]
        return torch.einsum("st,...tc->...sc", G, v)

    def one(self, v):
        """D on one spinor [V, 4, 3]."""
        v = v.reshape(self.L + (4, 3))
        out = self.diag * v
        for S, F in self.F:
            out = out + self._spin(S, self._colour(F, v))
        for mu in range(4):
            f = torch.roll(v, -1, mu)
            b = self._colour(self.U[mu].conj().transpose(-1, -2), v)
            b = torch.roll(b, 1, mu)
            if mu == 0:
                f[-1] *= -1.0
                b[0] *= -1.0
            f = self._colour(self.U[mu], f)
            out = out - 0.5 * (f - self._spin(self.g[mu], f) + b + self._spin(self.g[mu], b))
        return out.reshape(-1, 4, 3)

    @staticmethod
    def g5(v):
        return torch.cat((v[..., :2, :], -v[..., 2:, :]), -2)

    def dag(self, v):
        return self.g5(self.one(self.g5(v)))

    def solve(self, b, steps=5000):
        """D x = b by CG on the normal equations to rounding."""
        x, r = torch.zeros_like(b), self.dag(b)
        p, rr = r, torch.vdot(r.flatten(), r.flatten()).real
        stop = 1e-30 * rr
        for _ in range(steps):
            q = self.dag(self.one(p))
            a = rr / torch.vdot(p.flatten(), q.flatten()).real
            x, r = x + a * p, r - a * q
            new = torch.vdot(r.flatten(), r.flatten()).real
            if new <= stop:
                break
            p, rr = r + (new / rr) * p, new
        return x


class _Basis:
    """The block basis of Gaussian test vectors, orthonormal per block and
    chirality with positive diagonal R, [blocks, 2, 6 |B|, nv]."""

    def __init__(self, case, seed):
        self.case = case
        A = self.blocked(_spinors(case, seed, case["nv"], 4)).permute(1, 2, 3, 0).contiguous()
        for _ in range(3):
            R = torch.linalg.cholesky(torch.matmul(A.mH, A)).mH
            A = torch.linalg.solve_triangular(R, A, upper=True, left=False)
        self.A = A

    def blocked(self, v):  # [n, V, 4, 3] -> [n, blocks, 2, 6 |B|]
        L, b = _L(self.case), self.case["block"]
        y = [q // b for q in L]
        v = v.reshape(-1, y[0], b, y[1], b, y[2], b, y[3], b, 2, 6)
        return v.permute(0, 1, 3, 5, 7, 9, 2, 4, 6, 8, 10).reshape(v.shape[0], math.prod(y), 2, 6 * b ** 4)

    def unblocked(self, w):
        L, b = _L(self.case), self.case["block"]
        y = [q // b for q in L]
        w = w.reshape(-1, y[0], y[1], y[2], y[3], 2, b, b, b, b, 6)
        return w.permute(0, 1, 6, 2, 7, 3, 8, 4, 9, 5, 10).reshape(w.shape[0], math.prod(L), 4, 3)

    def restrict(self, v):  # [n, V, 4, 3] -> [n, blocks, 2 nv]
        return torch.einsum("yakc,nyak->nyac", self.A.conj(), self.blocked(v)).reshape(v.shape[0], -1, 2 * self.A.shape[-1])

    def prolong(self, c):
        c = c.reshape(c.shape[0], -1, 2, self.A.shape[-1])
        return self.unblocked(torch.einsum("yakc,nyac->nyak", self.A, c))


def exact(case, seed):
    what, n = case["what"], case["nrhs"]
    L = _L(case)
    if what == "dirac":
        D, v = _Dirac(case, seed), _spinors(case, seed, n)
        f = {"D": D.one, "Ddag": D.dag, "Q": lambda q: D.g5(D.one(q)), "DdagD": lambda q: D.dag(D.one(q))}[case["op"]]
        for r in range(n):
            v[r] = f(v[r].clone())
        return v
    if what == "project":
        P, v = _Basis(case, seed), _spinors(case, seed, n)
        c = torch.cat([P.restrict(v[r:r + 1]) for r in range(n)])
        for r in range(n):
            v[r] = P.prolong(c[r:r + 1])[0]
        return {"coarse": c, "fine": v}
    if what == "coarse":
        D, P = _Dirac(case, seed), _Basis(case, seed)
        nv = case["nv"]
        x = _complex_randn((n, _coarse_volume(case), 2 * nv), _gen(seed, 2))
        sign = torch.cat((torch.ones(nv), -torch.ones(nv))).to(x)
        out = []
        for r in range(n):
            c = x[r] * sign if case["op"] == "Ddag" else x[r]
            y = P.restrict(D.one(P.prolong(c[None])[0])[None])[0]
            out.append(y if case["op"] == "D" else y * sign)
        return torch.stack(out)
    if what == "contract":
        a = _spinors(case, seed, 3 * n, 2).reshape(n, 3, L[0], -1, 4, 3)
        b = _spinors(case, seed, n, 3).reshape(n, L[0], -1, 4, 3)
        g = _gammas()
        g5 = torch.diag(torch.tensor([1, 1, -1, -1], dtype=torch.complex128)).cuda()
        out = torch.zeros((n, L[0]), device="cuda", dtype=torch.complex128)
        for r in range(n):
            for k in range(3):
                t = torch.einsum("st,txyc->sxyc", g5 @ g[k + 1], b[r].permute(2, 0, 1, 3))
                out[r] += (a[r, k].conj() * t.permute(1, 2, 0, 3)).sum((1, 2, 3))
        return -out / (3.0 * L[1] * L[2] * L[3])
    if what == "solve" and _volume(case) * n <= 40000:
        D, b = _Dirac(case, seed), _spinors(case, seed, n, z2=True)
        x = torch.stack([D.solve(b[r]) for r in range(n)])
        return {"x": x, "x_coarse": None} if case["pieces"] else {"x": x}
    return None
