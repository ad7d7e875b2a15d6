"""The soft quantiser's backward in a graph, where a kernel of its own clears the sums whatever the size:
replayed with sums of an earlier replay in place, inputs written just ahead on the stream, and other calls
of the library in front of it and behind it in the graph."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 7, 2049, 100000, 786431, 786432, 1000003])
def test_replays(n):
    import paper_1908_05033_b200 as dsq
    gen = torch.Generator(device="cuda").manual_seed(n)
    x0, g0 = (torch.randn(n, device="cuda", generator=gen) for _ in range(2))
    x, g, gx, y, y2 = (torch.empty(n, device="cuda") for _ in range(5))
    sums = torch.full((3,), 1e30, dtype=torch.float64, device="cuda")
    args = (4, -1.0, 2.0, 0.2)

    def calls():
        dsq.dsq_soft_quantize_fwd(x, *args, out=y)
        dsq.dsq_soft_quantize_bwd(x, g, *args, out=gx, grad_params=sums)
        dsq.dsq_soft_quantize_fwd(gx, *args, out=y2)

    x.copy_(x0)
    g.copy_(g0)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        calls()
    torch.cuda.current_stream().wait_stream(side)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        calls()
    sums.fill_(float("nan"))
    got = []
    for i in range(6):
        torch.mul(x0, 1.0 + i, out=x)
        torch.mul(g0, 1.0 - 0.125 * i, out=g)
        graph.replay()
        got.append([t.clone() for t in (y, gx, y2, sums)])
    # (one binary64 addition a block, at most 600 of them, in any order; no term exceeds
    # 40 |g|: tanh, x - m and phi are bounded on [-1, 2])
    bound = 600 * 2.0 ** -52 * 40 * (float(g0.abs().sum()) * 1.01 + 1.0)
    for i in range(6):
        torch.cuda.synchronize()
        torch.mul(x0, 1.0 + i, out=x)
        torch.mul(g0, 1.0 - 0.125 * i, out=g)
        calls()
        for a, b in zip(got[i], (y, gx, y2)):
            assert torch.equal(a, b)
        assert float((got[i][3] - sums).abs().max()) <= bound
