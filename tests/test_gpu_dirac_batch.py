"""FP64 operator: a RHS gets the same bits alone (a warp per direction on small
calls) and in a batch that takes one thread per site."""
import numpy as np
import pytest

import synthetic
from gpu_util import to_device

pytestmark = pytest.mark.gpu


# 630 sites: 19.7 warps, the last one ragged; both time boundaries; extents 1 and 2
@pytest.mark.parametrize("L,nrhs,t_bc", [((5, 6, 7, 3), 21, -1), ((8, 8, 8, 8), 4, 1), ((2, 1, 3, 2), 1100, -1)])
def test_alone_and_in_a_batch(L, nrhs, t_bc):
    import torch
    import paper_2412_06347_gb300 as m
    ctx = m.Context(0)
    V = int(np.prod(L))
    assert V <= 12288 < V * nrhs
    g = m.mglma_gauge_load(ctx, L, synthetic.gauge_links(L, 0.3, 81), 0.13, 1.4, t_bc=t_bc)
    x = to_device(synthetic.random_spinors(L, nrhs, 82))
    for op in ("D", "DDAG", "Q", "DDAGD"):
        code = getattr(m, "MGLMA_OP_" + op)
        out, one = torch.zeros_like(x), torch.zeros_like(x)
        m.mglma_dirac_apply(ctx, g, code, nrhs, x, out, m.MGLMA_FP64)
        for r in range(nrhs):
            m.mglma_dirac_apply(ctx, g, code, 1, x[r], one[r], m.MGLMA_FP64)
        torch.cuda.synchronize()
        assert bool((out.abs() > 0).any())
        assert torch.equal(out, one), (op, (out - one).abs().max().item())
    m.mglma_gauge_free(g)
    ctx.close()
