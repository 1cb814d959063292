"""The contraction gives the same bits from the grid with a CTA per chunk of 1024
sites (a direct call) and from the one with a CTA per slice (a captured call)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,nrhs", [((3, 8, 8, 8), 2), ((2, 8, 8, 16), 1), ((3, 5, 15, 41), 2), ((4, 16, 16, 12), 3),
                                    ((2, 32, 32, 33), 2)])
def test_direct_and_captured(L, nrhs):
    import torch
    import paper_2412_06347_gb300 as m
    ctx = m.Context(0)
    gen = torch.Generator("cuda").manual_seed(11)

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
    assert bool((out[0].abs() > 0).all())
    assert torch.equal(out[0], out[1])
    ctx.close()
