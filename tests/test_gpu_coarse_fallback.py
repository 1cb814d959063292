"""The default coarse solver MINRES_EO where its even-odd form cannot run -- a
coarse grid with an odd extent, an operator stored in FP32 -- is MINRES on Q1:
the same iterates as MGLMA_COARSE_MINRES, bit for bit, in the preconditioner,
and the pieces reach their tolerance in the FP64 residual of the coarse
operator."""
import numpy as np
import pytest

import synthetic

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


# coarse grids 3x2x2x2, 3^4 (tensor cores, Nv 8), 1x2x2x2 (Nv 6: no tensor image), 2^4 stored in FP32
@pytest.mark.parametrize("L,block,nv,store", [
    ((12, 4, 4, 4), (4, 2, 2, 2), 8, "BF16"),
    ((6, 6, 6, 6), (2, 2, 2, 2), 8, "BF16"),
    ((4, 4, 4, 4), (4, 2, 2, 2), 6, "BF16"),
    ((4, 4, 4, 4), (2, 2, 2, 2), 8, "FP32"),
])
@pytest.mark.parametrize("graph", [0, 1])
def test_default_runs_as_minres(m, ctx, L, block, nv, store, graph):
    nrhs = 3
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 91), 0.122, 1.2)
    sub = m.mglma_subspace_build(ctx, g, block, nv, 5, 92, m.MGLMA_FP64)
    C = m.mglma_coarse_build(ctx, g, sub, getattr(m, "MGLMA_" + store))
    b = synthetic.random_spinors(L, nrhs, 93)
    xs, its, pieces = [], [], []
    for solver in (2, 1):  # MINRES_EO (the default), MINRES
        prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, coarse_solver=solver, graph=graph, tol=1e-11)
        x, xc = np.zeros_like(b), np.zeros_like(b)
        _, st = m.mglma_solve_batch(ctx, g, C, prm, [nrhs], b, x, xc)
        assert all(s["converged"] for s in st)
        xs.append(x)
        pieces.append(xc)
        its.append([(s["iterations"], s["coarse_iterations"]) for s in st])
    assert its[0] == its[1]
    assert np.array_equal(xs[0], xs[1]) and np.array_equal(pieces[0], pieces[1])
    # D1 X = R0 b for X = R0 psi1 (R0 T0 = 1): the residual the solve stops on
    n2, V1 = 2 * nv, int(np.prod([l // s for l, s in zip(L, block)]))
    X, b1, D1X = (np.zeros((nrhs, V1, n2), complex) for _ in range(3))
    m.mglma_restrict(ctx, sub, nrhs, pieces[0], X)
    m.mglma_restrict(ctx, sub, nrhs, b, b1)
    m.mglma_coarse_apply(ctx, C, nrhs, X, D1X)
    res = np.linalg.norm((b1 - D1X).reshape(nrhs, -1), axis=1) / np.linalg.norm(b1.reshape(nrhs, -1), axis=1)
    # tol / 10 asked for; T0 and R0 round X by about 2 n2 u |D1| / |D1^-1|, far below tol
    assert res.max() <= 1e-11, res
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
