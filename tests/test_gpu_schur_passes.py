"""Every pass of the even-odd stencil against the FP64 oracle's D restricted to
the parities, on half volumes that are no multiple of a warp and with extents 2.

Tolerances, u = 2^-24: a component goes through at most 160 FP32 roundings (two
sweeps of eight hops of ten roundings, two clover blocks), so a pass is within
160 u = 1e-5 of the operands' norm times |S| / |S x| (below 3 here); BF16 results
add half an ulp, 2^-9 per component.  Sums of a warp take 24 products per thread
and five additions, 32 roundings, of the magnitudes: 32 u sum |a||b|."""
import numpy as np
import pytest

import synthetic
from oracle import dirac as D
from schur_driver import from_half, load, parity_sites, to_half

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
TOL = 3 * 160 * U
KAPPA, CSW = 0.12, 1.2


@pytest.fixture(scope="module")
def m():
    import paper_2412_06347_gb300 as mod
    return mod


@pytest.fixture(scope="module")
def ctx(m):
    c = m.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def drv(m, tmp_path_factory):
    return load(m, tmp_path_factory.mktemp("schur"))


class Ref:
    """D in parity blocks on canonical fields, complex128."""

    def __init__(self, L, t_bc):
        self.L, self.t_bc = L, float(t_bc)
        self.links = synthetic.gauge_links(L, 0.25, 71)
        self.A = D.clover_matrix(self.links, KAPPA, CSW)
        self.Ai = np.linalg.inv(self.A.reshape(-1, 12, 12))
        self.ev, self.od = parity_sites(L)

    def full(self, h, sites):
        f = np.zeros((h.shape[0], int(np.prod(self.L)), 12), complex)
        f[:, sites] = h
        return f.reshape((h.shape[0],) + self.L + (4, 3))

    def D(self, h, src, dst):
        r = D.dirac(self.links, self.full(h, src), KAPPA, CSW, bc_t=self.t_bc, A=self.A)
        return r.reshape(h.shape[0], -1, 12)[:, dst]

    def oo_inv(self, h):
        return np.einsum("xij,nxj->nxi", self.Ai[self.od], h)

    def odd(self, xe):
        return self.oo_inv(self.D(xe, self.ev, self.od))

    def S(self, xe):
        return self.D(xe, self.ev, self.ev) - self.D(self.odd(xe), self.od, self.ev)


def close(got, ref, scale=None, tol=TOL):
    for r in range(ref.shape[0]):
        err = np.linalg.norm(got[r] - ref[r])
        assert err <= tol * np.linalg.norm((ref if scale is None else scale)[r]), (r, err)


def close_bf16(got, ref):
    # half an ulp of the rounded value, plus the FP32 error before rounding
    n = np.sqrt(np.mean(np.abs(ref) ** 2))
    for a, b in ((got.real, ref.real), (got.imag, ref.imag)):
        assert np.all(np.abs(a - b) <= 2.0 ** -8 * np.abs(b) + 20 * TOL * n)


@pytest.mark.parametrize("L,nrhs,t_bc", [((4, 6, 2, 10), 3, -1), ((2, 2, 4, 6), 2, 1), ((8, 4, 4, 4), 1, -1)])
def test_passes(m, ctx, drv, L, nrhs, t_bc):
    import torch
    f32, bf = torch.float32, torch.bfloat16
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 71), KAPPA, CSW, t_bc=t_bc)
    assert drv.ready(ctx, g)
    ref = Ref(L, t_bc)
    ev, od, Vh = ref.ev, ref.od, len(ref.ev)
    psi, phi, chi = (synthetic.random_spinors(L, nrhs, s) for s in (1, 2, 3))

    def new(dtype=f32):
        return torch.zeros((nrhs, 6, Vh, 4) if dtype == f32 else (nrhs, 3, Vh, 8), device="cuda", dtype=dtype)

    for dtype, prec in ((f32, m.MGLMA_FP32), (bf, m.MGLMA_BF16)):
        x = to_half(psi, ev, dtype)
        w = new()
        drv("odd", ctx, g, nrhs, x, prec, w)
        close(from_half(w), ref.odd(from_half(x)))
    x, b, bo = to_half(psi, ev, f32), to_half(phi, ev, f32), to_half(chi, od, f32)
    xr, br, bor = from_half(x), from_half(b), from_half(bo)
    Sx = ref.S(xr)
    drv("odd", ctx, g, nrhs, x, m.MGLMA_FP32, w)
    out = new()
    drv("apply", ctx, g, nrhs, w, x, out)
    close(from_half(out), Sx)
    drv("odd_solution", ctx, g, nrhs, None, bo, out)
    close(from_half(out), ref.oo_inv(bor))
    drv("odd_solution", ctx, g, nrhs, x, bo, out)
    close(from_half(out), ref.oo_inv(bor - ref.D(xr, ev, od)), scale=bor + ref.D(xr, ev, od))
    drv("prepare", ctx, g, nrhs, b, bo, out)
    close(from_half(out), br - ref.D(bor, od, ev))
    s = new(bf)
    drv("resid", ctx, g, nrhs, w, x, b, s, m.MGLMA_BF16)
    close_bf16(from_half(s), br - Sx)
    # the first MR step's t = S s and alpha = <t, s> / |t|^2 of the stored values
    drv("odd", ctx, g, nrhs, s, m.MGLMA_BF16, w)
    t, al = new(bf), torch.zeros((nrhs, 2), device="cuda")
    drv("dot", ctx, g, nrhs, w, s, t, m.MGLMA_BF16, al)
    sr, tr = from_half(s), from_half(t)
    close_bf16(tr, ref.S(sr))

    def alpha_ok(a, t_, s_):
        a = a.cpu().double().numpy()
        for r in range(nrhs):
            tt = np.vdot(t_[r], t_[r]).real
            want = np.vdot(t_[r], s_[r]) / tt
            assert abs(a[r, 0] + 1j * a[r, 1] - want) <= 4 * 32 * U * np.abs(t_[r] * s_[r]).sum() / tt

    alpha_ok(al, tr, sr)
    # t' = t - a S t, s' = s - a t
    drv("odd", ctx, g, nrhs, t, m.MGLMA_BF16, w)
    tn, sn, aln = new(bf), new(bf), torch.zeros((nrhs, 2), device="cuda")
    drv("mr", ctx, g, nrhs, w, t, tn, s, sn, m.MGLMA_BF16, al, aln)
    a = al.cpu().double().numpy()
    a = (a[:, 0] + 1j * a[:, 1])[:, None, None]
    close_bf16(from_half(tn), tr - a * ref.S(tr))
    close_bf16(from_half(sn), sr - a * tr)
    alpha_ok(aln, from_half(tn), from_half(sn))
    # the FGCR image with its dots: slot 0 with the residual, slots 1 to 3 with the earlier images
    W = torch.randn((3, nrhs, 6, Vh, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    drv("odd", ctx, g, nrhs, x, m.MGLMA_FP32, w)
    for k in range(4):
        nw = torch.zeros(nrhs, device="cuda", dtype=torch.float64)
        num, dots = (torch.zeros((3 * nrhs, 2), device="cuda", dtype=torch.float64) for _ in range(2))
        drv("gcr", ctx, g, nrhs, w, x, out, k, W, b, nw, num, dots)
        o = from_half(out)
        close(o, Sx)
        for r in range(nrhs):
            if k == 0:
                assert abs(nw[r].item() - np.vdot(o[r], o[r]).real) <= 32 * U * np.vdot(o[r], o[r]).real
                pairs = [(num[r], o[r], br[r])]
            else:
                pairs = [(dots[j * nrhs + r], from_half(W[j])[r], o[r]) for j in range(k)]
            for got, p, q in pairs:
                got = got.cpu().numpy()
                assert abs(got[0] + 1j * got[1] - np.vdot(p, q)) <= 2 * 32 * U * np.abs(p * q).sum()
    m.mglma_gauge_free(g)
