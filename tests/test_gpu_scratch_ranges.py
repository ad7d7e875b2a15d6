"""Requantiser ranges at the limits of binary32: the codes-only call, which has epilogues
of its own, gives the codes of the call that also returns fp32 (one general epilogue)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# the reciprocal of the step is infinite, denormal or zero, or the width overflows
RANGES = [(0.0, 1e-44), (0.0, 1e-38), (0.0, 4.3e-38), (0.0, 4.5e-38), (0.0, 3e38), (-1e-38, 1e-38),
          (-3e38, 3e38), (0.0, 1e-30), (0.0, 1e-23), (0.0, 1.0)]


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


def affine(c, rng):
    """Scales and biases that put results below, inside, on and above the range; a third
    of the channels give 0 throughout."""
    g = torch.Generator(device="cuda").manual_seed(c)
    width = min(rng[1] - rng[0], 1e36)
    scale = torch.randn(c, device="cuda", generator=g) * (width / 100)
    bias = torch.randn(c, device="cuda", generator=g) * (width / 4)
    scale[::3], bias[::3] = 0, 0
    return scale, bias


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("stride", [1, 2])
def test_depthwise(dsq, bits, stride):
    C, shape = 40, (2, 9, 7, 40)
    torch.manual_seed(bits)
    act = dsq.dsq_quantize_act(torch.rand(shape, device="cuda") * 6, bits, 0.0, 6.0)
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(torch.randn(C, 3, 3, device="cuda") * 0.3, bits, -1.0, 1.0, ws,
                                      depthwise=True, stride=stride, pad=1)
    for rng in RANGES:
        scale, bias = affine(C, rng)
        both = [dsq.dsq_dwconv2d(act, shape, (bits, 0.0, 6.0), blob, conv, scale, bias, w_offset=0.5,
                                 requant=(bits,) + rng, want_f32=f32)[0] for f32 in (True, False)]
        assert torch.equal(*both), rng


# (hook, N, H, W, Cin, Cout, k, stride): the kernel for little work, the window kernel on
# transposed and plain tiles, the 1x1 kernel, the im2col kernel
DENSE = [(1, 1, 6, 5, 64, 40, 3, 1), (1, 1, 6, 5, 40, 72, 1, 1), (3, 2, 9, 7, 64, 40, 3, 1),
         (3, 1, 8, 8, 128, 136, 3, 1), (4, 1, 8, 8, 128, 136, 3, 1), (3, 2, 9, 7, 40, 72, 1, 1),
         (3, 2, 9, 7, 40, 72, 1, 2), (0, 2, 9, 7, 64, 40, 3, 2)]


@pytest.mark.parametrize("res_rng", [None, (-1.0, 2.0), (-3e38, 3e38), (0.0, 1e-44)])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("case", DENSE)
def test_dense(dsq, case, res_rng, bits):
    """... with residual ranges whose width overflows or whose step is a denormal number."""
    hook, n, h, w, ci, co, k, stride = case
    torch.manual_seed(bits)
    act = dsq.dsq_quantize_act(torch.rand(n, h, w, ci, device="cuda") * 6, bits, 0.0, 6.0)
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(torch.randn(co, k, k, ci, device="cuda") * 0.05, bits, -0.1, 0.1,
                                      ws, stride=stride, pad=k // 2)
    kw = {}
    if res_rng:
        ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
        codes = torch.randint(0, 2 ** bits, (n * ho * wo, co), device="cuda", dtype=torch.int8)
        kw = dict(residual=dsq.dsq_pack_codes(codes, bits), residual_q=(bits,) + res_rng)
    dsq.dsq_set_conv3_window(hook)
    try:
        for rng in RANGES:
            scale, bias = affine(co, rng)
            both = [dsq.dsq_conv2d(act, (n, h, w, ci), (bits, 0.0, 6.0), blob, conv, scale, bias, ws,
                                   w_offset=0.5, requant=(bits,) + rng, want_f32=f32, **kw)[0]
                    for f32 in (True, False)]
            assert torch.equal(*both), rng
    finally:
        dsq.dsq_set_conv3_window(1)
