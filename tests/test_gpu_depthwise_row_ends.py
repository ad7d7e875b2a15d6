"""Depthwise convolution on 3-bit rows that end inside their last unit of eight channels
(and their neighbours that do not): every code, sum and fp32 result against the oracle,
nothing written behind the last row and no row's start disturbed by the one before."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from test_gpu_conv import dw_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


CHANNELS = [40, 41, 42, 43, 81, 84, 85, 169, 170, 171, 298]


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("c", CHANNELS)
def test_row_ends(dsq, c, stride):
    dw_case(dsq, 2, 9, 14, c, stride, 3, 0.5)
    dw_case(dsq, 2, 9, 14, c, stride, 3, 0.3, residual=stride == 1)
    # codes alone, into the front of a larger buffer; inputs at its very end
    shape, pitch, bits = (2, 9, 14, c), dsq.dsq_row_pitch(c, 3), 3
    gen = np.random.default_rng(c)
    q = torch.from_numpy(gen.integers(0, 8, (2 * 9 * 14, c)).astype(np.int8)).cuda()
    act = dsq.dsq_pack_codes(q, bits)
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(torch.randn(c, 3, 3, device="cuda"), bits, -1.0, 1.0, ws,
                                      depthwise=True, stride=stride, pad=1)
    args = (act, shape, (bits, 0.0, 6.0), blob, conv, torch.full((c,), 0.05, device="cuda"),
            torch.full((c,), 1.0, device="cuda"))
    want, _, _ = dsq.dsq_dwconv2d(*args, requant=(bits, 0.0, 6.0), want_f32=True)
    buf = torch.full((want.numel() + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    out = buf[:want.numel()].view(want.shape)
    dsq.dsq_dwconv2d(*args, requant=(bits, 0.0, 6.0), out_codes=out)
    assert torch.equal(out, want)
    assert (buf[want.numel():] == 0xA5).all()
