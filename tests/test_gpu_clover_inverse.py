"""Inverse clover blocks that need their pivoting (no mass, strong clover term), and
blocks that have no inverse (no mass, no clover term).

The Schur operator with such blocks against numpy's inverse in FP64: a 6x6
elimination with partial pivoting loses about 6 cond u per block; 50 max cond u,
u = 2^-53, is asked for.  Without an inverse the multigrid solve takes the
full-lattice system."""
import numpy as np
import pytest

import synthetic
from oracle import dirac as D
from schur_driver import load, parity_sites

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import paper_2412_06347_gb300 as mod
    return mod


@pytest.fixture(scope="module")
def ctx(m):
    c = m.Context(0)
    yield c
    c.close()


def test_pivoted_blocks(m, ctx):
    L, kappa, csw, n = (4, 6, 4, 4), 1e12, 1.4, 2
    U = synthetic.gauge_links(L, 0.9, 71)
    A = D.clover_matrix(U, kappa, csw)
    ev, od = parity_sites(L)
    Ao = A.reshape(-1, 12, 12)[od]
    blocks = np.concatenate([Ao[:, :6, :6], Ao[:, 6:, 6:]])
    assert np.mean(np.abs(blocks[:, :, 0]).argmax(axis=1) != 0) > 0.2  # row exchanges from the first column on
    cond = np.linalg.cond(blocks).max()
    x = synthetic.random_spinors(L, n, 5)
    f = x.reshape(n, -1, 12).copy()
    f[:, od] = 0

    def apply(v):
        return D.dirac(U, v.reshape(x.shape), kappa, csw, A=A).reshape(n, -1, 12)

    Dx = apply(f)
    w = np.zeros_like(f)
    w[:, od] = np.einsum("xij,nxj->nxi", np.linalg.inv(Ao), Dx[:, od])
    Hw = apply(w)[:, ev]
    S = Dx[:, ev] - Hw
    g = m.mglma_gauge_load(ctx, L, U, kappa, csw)
    out = np.zeros_like(x)
    m.mglma_dirac_apply(ctx, g, m.MGLMA_OP_SCHUR, n, x, out, m.MGLMA_FP64)
    got = out.reshape(n, -1, 12)
    assert np.linalg.norm(got[:, ev] - S) <= 50 * cond * 2.0 ** -53 * np.linalg.norm(Hw)
    m.mglma_gauge_free(g)


def test_singular_blocks(m, ctx, tmp_path):
    L, n = (2, 4, 4, 4), 2
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.3, 71), np.inf, 0.0)
    assert not load(m, tmp_path).ready(ctx, g)
    # blocks of one site and all six components of each chirality: the coarse
    # correction is the whole operator, so the hops alone converge
    sub = m.mglma_subspace_load(ctx, g, (1, 1, 1, 1), 6, np.ascontiguousarray(synthetic.random_spinors(L, 6, 5)),
                                m.MGLMA_FP32)
    C = m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)
    b = synthetic.random_spinors(L, n, 73)
    x, Dx = np.zeros_like(b), np.zeros_like(b)
    prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, tol=1e-8, coarse_max_iter=400)
    _, st = m.mglma_solve_batch(ctx, g, C, prm, [n], b, x)
    assert all(s["converged"] for s in st)
    m.mglma_dirac_apply(ctx, g, m.MGLMA_OP_D, n, x, Dx, m.MGLMA_FP64)
    assert np.linalg.norm(b - Dx) <= 1.01e-8 * np.linalg.norm(b)
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
