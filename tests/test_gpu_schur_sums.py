"""The dots of the even-odd passes on a lattice whose CTAs take four runs of 32
sites: FP32 sums stay within one run.  On free links a constant field gives the
same value at every site, so a factor of 2^20, -2^20, 1, 1 on the four runs
cancels exactly in FP64 sums of the runs and leaves 32 u of the rest; carried in
FP32 from run to run the large terms leave u 2^20 = 6 % behind."""
import numpy as np
import pytest

from schur_driver import from_half, load

pytestmark = pytest.mark.gpu
U = 2.0 ** -24
L = (32, 16, 32, 32)  # 2^18 half-lattice sites


def test_runs_are_added_in_fp64(tmp_path):
    import torch
    import paper_2412_06347_gb300 as m
    drv = load(m, tmp_path)
    ctx = m.Context(0)
    g = m.mglma_gauge_random(ctx, L, 0.0, 1, 0.12, 0.0, t_bc=1)
    assert drv.ready(ctx, g)
    Vh, n = int(np.prod(L)) // 2, 2
    c = torch.tensor([2.0 ** 20, -(2.0 ** 20), 1.0, 1.0], device="cuda")[(torch.arange(Vh, device="cuda") // 32) % 4]
    v = torch.randn((n, 6, 1, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    x = v.expand(n, 6, Vh, 4).contiguous()
    w, out = torch.zeros_like(x), torch.zeros_like(x)
    nw = torch.zeros(n, device="cuda", dtype=torch.float64)
    num, dots = (torch.zeros((3 * n, 2), device="cuda", dtype=torch.float64) for _ in range(2))
    drv("odd", ctx, g, n, x, m.MGLMA_FP32, w)
    drv("apply", ctx, g, n, w, x, out)
    assert bool((out == out[:, :, :1]).all())
    r = out * c[None, None, :, None]
    drv("gcr", ctx, g, n, w, x, out, 0, r, r, nw, num, dots)
    o2 = out.double().square().sum(dim=(1, 2, 3))
    assert bool(((nw - o2).abs() <= 32 * U * o2).all())
    assert bool(((num[:n, 0] - o2 / 2).abs() <= 32 * U * o2).all()), (num[:n, 0] / o2).tolist()
    # MR step with step length zero: t' = t, s' = s and the next length is <t, s> / |t|^2
    t = torch.randn((n, 3, 1, 8), device="cuda", generator=torch.Generator("cuda").manual_seed(4)).to(torch.bfloat16)
    t = t.expand(n, 3, Vh, 8).contiguous()
    s = t * c.to(torch.bfloat16)[None, None, :, None]
    tn, sn = torch.zeros_like(t), torch.zeros_like(s)
    al, aln = torch.zeros((n, 2), device="cuda"), torch.zeros((n, 2), device="cuda")
    drv("mr", ctx, g, n, w, t, tn, s, sn, m.MGLMA_BF16, al, aln)
    assert torch.equal(tn, t) and torch.equal(sn, s)
    assert bool(((aln[:, 0] - 0.5).abs() <= 2 * 32 * U).all()), aln.tolist()
    m.mglma_gauge_free(g)
    ctx.close()
