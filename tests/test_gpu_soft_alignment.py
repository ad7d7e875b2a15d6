"""The soft quantiser's two kernels on arrays that start 0, 16 or both offsets from a
32-byte boundary: the vector loop's head and tail give the bits that aligned arrays
give, element by element, and the three sums agree to the order of addition."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ox,og", [(4, 4), (4, 0), (0, 4)])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 11, 12, 13, 2052, 70001])
def test_soft_quantize_alignment(ox, og, n):
    import paper_1908_05033_b200 as dsq
    torch.manual_seed(n)
    x = torch.randn(n, device="cuda") * 1.2
    g = torch.randn(n, device="cuda")

    def at(v, o):
        buf = torch.zeros(n + 12, device="cuda")
        buf[o:o + n] = v
        return buf, buf[o:o + n]

    quant = (4, -1.0, 2.0, 0.2)
    y = dsq.dsq_soft_quantize_fwd(x, *quant)
    gx, gp = dsq.dsq_soft_quantize_bwd(x, g, *quant)
    _, xs = at(x, ox)
    _, gs = at(g, og)
    buf, out = at(torch.zeros(n, device="cuda"), og)
    dsq.dsq_soft_quantize_fwd(xs, *quant, out=out)
    assert torch.equal(out, y)
    dsq.dsq_soft_quantize_bwd(xs, gs, *quant, out=out, grad_params=(p := torch.empty_like(gp)))
    assert torch.equal(out, gx)
    torch.testing.assert_close(p, gp, rtol=1e-5, atol=1e-5)
    buf[og:og + n] = 0
    assert not buf.any()                       # nothing written beside the array
