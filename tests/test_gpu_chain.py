"""Kernels that begin while the one before drains (csrc/launch_util.cuh): a chain
of operator applications, each reading what the one before wrote, gives the same
bits queued at once, captured in a graph, across streams, and one at a time."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,N", [(2, 31), (2, 243), (2, 729), (3, 27), (3, 41)])
@pytest.mark.parametrize("dtype", [torch.complex64, torch.complex128])
def test_chain_matches_one_at_a_time(d, N, dtype):
    import paper_1412_2033_gb300 as g
    ctx = g.Context.from_microstructure(W.centred_disk(N) if d == 2 else W.centred_sphere(N))
    x0 = torch.randn(ctx.field_shape, dtype=dtype, device="cuda", generator=torch.Generator("cuda").manual_seed(N))
    bufs = [torch.empty_like(x0) for _ in range(3)]

    def chain(stop=lambda k: None):
        x = x0
        for k in range(12):
            y, z = bufs[2 * k % 3], bufs[(2 * k + 1) % 3]   # written while its last reader may still be draining
            ctx.matvec(x, kind=k % 2, out=y)
            y.mul_(1e-4)                       # another library's kernel in between
            ctx.matvec(y, kind=k % 2, out=z)
            x = z
            stop(k)
        return x.clone()

    want = chain(lambda k: torch.cuda.synchronize())
    torch.cuda.synchronize()
    assert torch.isfinite(torch.view_as_real(want)).all()
    for _ in range(3):
        assert torch.equal(chain(), want)

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        y = chain()
    torch.cuda.current_stream().wait_stream(side)
    z = ctx.matvec(y)                          # the other stream reads it
    assert torch.equal(y, want) and torch.equal(z, ctx.matvec(want))

    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = chain()
    for _ in range(2):
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
