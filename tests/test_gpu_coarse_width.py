"""The RHS width tuned for the coarse operator does not change the even-odd coarse
solve: its iterates are the same bits for every choice, up to 32 RHS in one tile."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [2, 8, 9, 16, 17, 32, 33])
def test_tuned_width_leaves_the_solve_alone(nrhs):
    import paper_2412_06347_gb300 as m
    L, block, nv = (8, 4, 4, 4), (2, 2, 2, 2), 8
    ctx = m.Context(0)
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 71), 0.12, 1.2)
    sub = m.mglma_subspace_build(ctx, g, block, nv, 5, 72, m.MGLMA_FP32)
    C = m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)
    b = synthetic.random_spinors(L, nrhs, 73)
    prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, autotune=0)
    xs, its = [], []
    for width in (None, 8, 16, 32):
        if width:
            m.mglma_autotune_set(ctx, 1, nrhs, width)
        x = np.zeros_like(b)
        _, st = m.mglma_solve_batch(ctx, g, C, prm, [nrhs], b, x)
        assert all(s["converged"] for s in st)
        xs.append(x)
        its.append([s["coarse_iterations"] for s in st])
    for x, i in zip(xs[1:], its[1:]):
        assert i == its[0] and np.array_equal(x, xs[0])
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
    ctx.close()
