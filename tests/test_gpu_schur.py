"""The multigrid solve's FP32 system: the even-odd Schur system when every
extent is even, the full lattice otherwise.  One defect-correction cycle must
reach the FP32 target it was given in the FP64 residual of the full system
(an error of the parity-split stencil, its reconstruction or the smoother's
grouped update would leave it far above), on lattices whose half volume is no
multiple of a warp, with extents 2, with the periodic time boundary and for
smoother lengths on both sides of a group of steps."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

TOL = 1e-5  # one cycle: above inner_tol = 3e-6 and FP32 rounding of e


@pytest.fixture(scope="module")
def m():
    import paper_2412_06347_gb300 as mod
    return mod


@pytest.fixture(scope="module")
def ctx(m):
    c = m.Context(0)
    yield c
    c.close()


def solve(m, ctx, L, block, nrhs, nu, t_bc, tol, nv=4):
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.25, 71), 0.12, 1.2, t_bc=t_bc)
    sub = m.mglma_subspace_build(ctx, g, block, nv, 5, 72, m.MGLMA_FP32)
    C = m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)
    b = synthetic.random_spinors(L, nrhs, 73)
    x = np.zeros_like(b)
    prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, tol=tol, nu=nu)
    _, st = m.mglma_solve_batch(ctx, g, C, prm, [nrhs], b, x)
    Dx = np.zeros_like(b)
    m.mglma_dirac_apply(ctx, g, m.MGLMA_OP_D, nrhs, x, Dx, m.MGLMA_FP64)
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)
    res = np.linalg.norm((b - Dx).reshape(nrhs, -1), axis=1) / np.linalg.norm(b.reshape(nrhs, -1), axis=1)
    return st, res


@pytest.mark.parametrize("L,block,nrhs,t_bc", [
    ((8, 4, 4, 4), (2, 2, 2, 2), 1, -1),
    ((4, 6, 2, 10), (2, 3, 1, 5), 3, -1),    # half volume 240 = 7.5 warps
    ((2, 2, 4, 6), (1, 1, 2, 3), 2, 1),      # extents 2: both neighbours coincide; half volume 48
    ((16, 12, 16, 22), (4, 4, 4, 11), 9, -1),
    ((6, 3, 4, 4), (3, 3, 2, 2), 2, -1),     # an odd extent: the full-lattice system
])
def test_one_cycle_reaches_its_target(m, ctx, L, block, nrhs, t_bc):
    st, res = solve(m, ctx, L, block, nrhs, 7, t_bc, TOL)
    assert all(s["outer"] == 1 and s["converged"] for s in st), st
    assert res.max() <= TOL, res
    assert max(abs(s["residual"] - r) for s, r in zip(st, res)) <= 1e-3 * TOL


@pytest.mark.parametrize("nu", [1, 2, 8, 9, 18])  # 1, 1, 4, 5 and 9 steps on S in groups of four
def test_smoother_lengths(m, ctx, nu):
    st, res = solve(m, ctx, (8, 4, 4, 4), (2, 2, 2, 2), 2, nu, -1, 1e-10)
    assert all(s["converged"] and s["outer"] <= 3 for s in st), st
    assert res.max() <= 1e-10, res


def test_large_half_volume(m, ctx):
    # 2^18 half-lattice sites and more: several site blocks per CTA
    st, res = solve(m, ctx, (36, 16, 32, 32), (4, 4, 4, 4), 2, 7, -1, TOL)
    assert all(s["outer"] == 1 for s in st), st
    assert res.max() <= TOL, res


# 8 or more RHS take R0 / T0 of the even sites on the tensor cores where half a
# block fits them (64 / 128 sites), fewer RHS go through full fields: the same
# preconditioner to BF16 rounding of the transfers
@pytest.mark.parametrize("L,block", [
    ((8, 8, 8, 8), (4, 4, 4, 4)),     # 128 even sites per block
    ((4, 8, 8, 8), (2, 4, 4, 4)),     # 64: R0 on half fields, T0 on full ones
    ((8, 4, 16, 8), (4, 4, 8, 4)),    # 256
    ((6, 8, 8, 16), (3, 4, 4, 8)),    # odd side: block parities alternate; 192
    ((8, 8, 16, 6), (4, 4, 8, 3)),    # pairs along direction 2
    ((8, 16, 6, 6), (4, 8, 3, 3)),    # pairs along direction 1; 144 is no multiple of 64
])
def test_transfers_of_the_even_sites(m, ctx, L, block):
    many, res = solve(m, ctx, L, block, 9, 7, -1, TOL, nv=8)
    few, _ = solve(m, ctx, L, block, 2, 7, -1, TOL, nv=8)
    assert all(s["outer"] == 1 for s in many) and res.max() <= TOL
    assert max(abs(a["iterations"] - b["iterations"]) for a, b in zip(many, few)) <= 1, (many[:2], few)
