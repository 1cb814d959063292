"""The even-odd smoother keeps its fields in FP32 where the full-lattice one does:
for one step on D (nu = 1) and where a staged stencil tile (which has no fused
steps) was set.  Its passes in FP32 against the oracle (tolerances of
test_gpu_schur_passes), and the choice as seen in a solve: nu = 1 and nu = 2 are
both one step on S, so they differ in the fields' precision alone."""
import numpy as np
import pytest

import synthetic
from schur_driver import from_half, load, to_half
from test_gpu_schur_passes import CSW, KAPPA, U, Ref, close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nrhs,t_bc", [((4, 6, 2, 10), 3, -1), ((2, 2, 4, 6), 2, 1)])
def test_fp32_passes(L, nrhs, t_bc, tmp_path):
    import torch
    import paper_2412_06347_gb300 as m
    ctx = m.Context(0)
    drv = load(m, tmp_path)
    f32, prec = torch.float32, m.MGLMA_FP32
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 71), KAPPA, CSW, t_bc=t_bc)
    assert drv.ready(ctx, g)
    ref = Ref(L, t_bc)
    x, b = (to_half(synthetic.random_spinors(L, nrhs, s), ref.ev, f32) for s in (1, 2))
    w, s, t, tn, sn = (torch.zeros_like(x) for _ in range(5))
    al, aln = torch.zeros((nrhs, 2), device="cuda"), torch.zeros((nrhs, 2), device="cuda")

    def alpha_ok(a, t_, s_):
        a = a.cpu().double().numpy()
        for r in range(nrhs):
            tt = np.vdot(t_[r], t_[r]).real
            assert abs(a[r, 0] + 1j * a[r, 1] - np.vdot(t_[r], s_[r]) / tt) <= 4 * 32 * U * np.abs(t_[r] * s_[r]).sum() / tt

    drv("odd", ctx, g, nrhs, x, prec, w)
    drv("resid", ctx, g, nrhs, w, x, b, s, prec)
    sr = from_half(s)
    close(sr, from_half(b) - ref.S(from_half(x)))
    drv("odd", ctx, g, nrhs, s, prec, w)
    drv("dot", ctx, g, nrhs, w, s, t, prec, al)
    tr = from_half(t)
    close(tr, ref.S(sr))
    alpha_ok(al, tr, sr)
    drv("odd", ctx, g, nrhs, t, prec, w)
    drv("mr", ctx, g, nrhs, w, t, tn, s, sn, prec, al, aln)
    a = al.cpu().double().numpy()
    a = (a[:, 0] + 1j * a[:, 1])[:, None, None]
    close(from_half(tn), tr - a * ref.S(tr), scale=tr)
    close(from_half(sn), sr - a * tr, scale=sr)
    alpha_ok(aln, from_half(tn), from_half(sn))
    m.mglma_gauge_free(g)
    ctx.close()


def test_choice_in_a_solve():
    import paper_2412_06347_gb300 as m
    L, n = (8, 4, 4, 4), 2
    ctx = m.Context(0)
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 71), 0.12, 1.2)
    sub = m.mglma_subspace_build(ctx, g, (2, 2, 2, 2), 4, 5, 72, m.MGLMA_FP32)
    C = m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)
    b = synthetic.random_spinors(L, n, 73)

    plain, staged = m.dslash32_tile_code(1, 1), m.dslash32_staged_code(4)

    def solve(nu, tile):
        m.mglma_autotune_set(ctx, 0, n, tile)
        x = np.zeros_like(b)
        _, st = m.mglma_solve_batch(ctx, g, C, m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, nu=nu), [n], b, x)
        assert all(s["converged"] for s in st)
        return x

    for nu in (1, 2, 7):
        # a staged tile: FP32; any other: BF16 from two steps on
        assert np.array_equal(solve(nu, plain), solve(nu, staged)) == (nu == 1)
    assert np.array_equal(solve(1, plain), solve(2, staged)) and not np.array_equal(solve(1, plain), solve(2, plain))
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
    ctx.close()
