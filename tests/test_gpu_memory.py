"""Device memory of the multigrid solve and of the server: a solve with room for
the full-lattice form but not for the even-odd stencil's copies and fields takes
the former, and the bytes the server charges per slot are those it takes."""
import threading
import time

import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def m():
    import paper_2412_06347_gb300 as mod
    return mod


def setup(m, ctx, L):
    g = m.mglma_gauge_random(ctx, L, 0.2, 91, 0.12, 1.2)
    sub = m.mglma_subspace_build(ctx, g, (4, 4, 4, 4), 8, 3, 92, m.MGLMA_FP32)
    return g, sub, m.mglma_coarse_build(ctx, g, sub, m.MGLMA_BF16)


def free_all(m, g, sub, C):
    m.mglma_coarse_free(C)
    m.mglma_subspace_free(sub)
    m.mglma_gauge_free(g)


# bytes per site of one RHS with device buffers: 1152 of double-float copies, 576 of
# FP64 fields, then 1200 of FP32 fields on the full lattice, or 576 of copies and
# 1056 of fields in the even-odd form
@pytest.mark.parametrize("per_site", [3700, 3130])
def test_solve_in_what_room_there_is(m, per_site):
    import torch
    L = (32, 32, 32, 32)
    V = int(np.prod(L))
    ctx, solver = m.Context(0), m.Context(0)  # the second one's pool holds nothing yet
    g, sub, C = setup(m, ctx, L)
    c = torch.zeros((1, V // 256, 16), device="cuda", dtype=torch.complex128)
    m.mglma_coarse_apply(ctx, C, 1, c, torch.zeros_like(c), op=m.MGLMA_OP_SCHUR)  # forms the coarse inverses
    gen = torch.Generator("cuda").manual_seed(5)
    b = torch.view_as_complex(torch.randn((1,) + L + (4, 3, 2), device="cuda", dtype=torch.float64, generator=gen))
    x, Dx = torch.zeros_like(b), torch.zeros_like(b)
    prm = m.mglma_solve_params_default(m.MGLMA_SOLVER_MG, tol=1e-9)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    fill, step = [], 8 << 30
    while step >= 4 << 20:  # leave per_site V bytes and what is left of 4 MB
        while torch.cuda.mem_get_info()[0] - step >= per_site * V:
            fill.append(torch.empty(step, device="cuda", dtype=torch.uint8))
        step //= 2
    try:
        _, st = m.mglma_solve_batch(solver, g, C, prm, [1], b, x)
    finally:
        del fill
        torch.cuda.empty_cache()
    assert st[0]["converged"]
    m.mglma_dirac_apply(ctx, g, m.MGLMA_OP_D, 1, x, Dx, m.MGLMA_FP64)
    torch.cuda.synchronize()
    assert ((b - Dx).abs().square().sum() / b.abs().square().sum()).sqrt().item() <= 1.01e-9
    free_all(m, g, sub, C)
    solver.close()
    ctx.close()


def test_server_charges_what_a_slot_takes(m):
    import torch
    L = (32, 16, 16, 16)
    ctx = m.Context(0)
    g, sub, C = setup(m, ctx, L)
    gen = torch.Generator("cuda").manual_seed(6)
    b = torch.view_as_complex(torch.randn((24,) + L + (4, 3, 2), device="cuda", dtype=torch.float64, generator=gen))
    x = torch.zeros_like(b)
    low, stats = {}, {}
    torch.cuda.synchronize()
    for slots in (8, 8, 24):  # the first run forms what stays
        seen, stop = [], threading.Event()

        def watch():
            while not stop.is_set():
                seen.append(torch.cuda.mem_get_info()[0])
                time.sleep(0.002)

        t = threading.Thread(target=watch)
        t.start()
        stats[slots], res = m.mglma_serve(ctx, [(g, C)], [dict(lattice=0, b=b[:slots], x=x[:slots], arrival=0.0)],
                                          max_slots=slots)
        stop.set()
        t.join()
        assert res[0]["status"] == 0 and stats[slots]["slots"][0] == slots
        low[slots] = min(seen)
    took = (low[8] - low[24]) / 16
    charged = stats[24]["slot_bytes"][0]
    assert 0.85 * charged <= took <= 1.1 * charged, (took, charged)
    free_all(m, g, sub, C)
    ctx.close()
