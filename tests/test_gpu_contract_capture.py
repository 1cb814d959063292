"""The contraction inside a stream capture (one CTA per slice, no workspace)
against the direct call (one CTA per chunk of 1024 sites, partial sums): the
same products in the same order up to how a chunk's scaled sum is rounded.

Tolerance: each of the nc chunk sums c_i enters either as fl(scale c_i) or fused
into the running sum, and both sums take nc additions, so the two differ by at
most 4 nc u sum_i |scale c_i|, u = 2^-53, and |scale c_i| is at most the mean
over the slice of |a||b| per site (Cauchy-Schwarz over the site's components)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nrhs", [((3, 8, 8, 8), 2), ((2, 8, 8, 16), 1), ((3, 5, 15, 41), 2), ((4, 16, 16, 12), 3)])
def test_contract_under_capture(L, nrhs):
    import torch
    import paper_2412_06347_gb300 as m
    ctx = m.Context(0)
    gen = torch.Generator("cuda").manual_seed(7)

    def field(n):
        v = torch.randn((n,) + tuple(L) + (4, 3, 2), device="cuda", dtype=torch.float64, generator=gen)
        return torch.view_as_complex(v).contiguous()

    a, b = field(3 * nrhs), field(nrhs)
    out = torch.zeros((2, nrhs, L[0]), device="cuda", dtype=torch.complex128)
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    m.mglma_contract(ctx, L, nrhs, a, b, out[0], stream=stream)
    stream.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        m.mglma_contract(ctx, L, nrhs, a, b, out[1], stream=stream)
    graph.replay()
    torch.cuda.synchronize()
    slice_ = L[1] * L[2] * L[3]
    nc = (slice_ + 1023) // 1024
    an = a.abs().square().sum(dim=(-1, -2)).sqrt().view(nrhs, 3, L[0], slice_)
    bn = b.abs().square().sum(dim=(-1, -2)).sqrt().view(nrhs, 1, L[0], slice_)
    bound = 4 * nc * 2.0 ** -53 * (an * bn).sum(dim=(1, 3)) / (3.0 * slice_)
    assert bool(((out[1] - out[0]).abs() <= bound).all())
    assert bool((out[0].abs() > 0).all())
    ctx.close()
