"""The coarse-space piece of a RHS does not depend on its batch: bit for bit the
same alone and with RHS that need another cycle of the FP64 coarse solve, or
whose norm overflows.  The operator is tuned so that cycles repeat: its mass is
shifted until the smallest real eigenvalue of D1 is delta (the shift moves every
eigenvalue by the same amount, the basis being fixed and orthonormal), and half
the sources are images D1 c of random coarse fields, whose solutions lack the
large component along that eigenvector."""
import numpy as np
import pytest

import synthetic
from oracle import multigrid as MG

pytestmark = pytest.mark.gpu

L, BLK, NV, CSW, KAPPA = (4, 4, 4, 4), (2, 2, 2, 2), 8, 1.2, 0.12


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
def problem():
    U = synthetic.gauge_links(L, 0.25, 91)
    vecs = np.ascontiguousarray(synthetic.random_spinors(L, NV, 5))
    D1 = MG.dense_coarse(MG.coarse_operator(U, MG.build_basis(vecs, L, BLK), KAPPA, CSW, BLK), (2, 2, 2, 2))
    w = np.linalg.eigvals(D1)
    lam = w[np.abs(w.imag) < 1e-9].real.min()
    return U, vecs, lam


@pytest.mark.parametrize("delta,tol,nrhs", [(1e-3, 1e-13, 16), (1e-3, 3e-13, 5), (0.6, 1e-11, 16)])
def test_piece_alone_and_in_a_batch(m, ctx, problem, delta, tol, nrhs):
    U, vecs, lam = problem
    g = m.mglma_gauge_load(ctx, L, U, 1 / (2 * (1 / (2 * KAPPA) - lam + delta)), CSW)
    sub = m.mglma_subspace_load(ctx, g, BLK, NV, vecs, m.MGLMA_FP64)
    C = m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)
    b = synthetic.random_spinors(L, nrhs, 93)
    c = np.ascontiguousarray(synthetic.random_spinors(L, nrhs, 94).reshape(nrhs, -1)[:, :256].reshape(nrhs, 16, 16))
    D1c, e = np.zeros_like(c), np.zeros_like(b)
    m.mglma_coarse_apply(ctx, C, nrhs, c, D1c)
    m.mglma_prolong(ctx, sub, nrhs, D1c, e)
    b[::2] = e[::2]
    if delta == 0.6:
        b[2] *= 1e200  # |b|^2 overflows: this one is left out, the others are not
    psi = np.zeros((1,) + b.shape, complex)
    m.mglma_pieces(ctx, g, [C], nrhs, b, psi, tol=tol)
    for r in range(nrhs):
        if delta == 0.6 and r == 2:
            continue
        one = np.zeros((1, 1) + b.shape[1:], complex)
        m.mglma_pieces(ctx, g, [C], 1, b[r:r + 1], one, tol=tol)
        assert np.abs(one).max() > 0
        assert np.array_equal(one[0, 0], psi[0, r]), (r, np.abs(one[0, 0] - psi[0, r]).max())
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
