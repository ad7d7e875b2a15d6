"""Requantiser ranges at the limits of binary32: the codes-only call, which has epilogues
of its own, gives the codes of the call that also returns fp32 (one general epilogue)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# the reciprocal of the step is infinite, denormal or zero, or the width overflows
RANGES = [(0.0, 1e-44), (0.0, 1e-38), (0.0, 4.3e-38), (0.0, 4.5e-38), (0.0, 3e38), (-1e-38, 1e-38),
          (-3e38, 3e38), (0.0, 1.0)]


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


@pytest.mark.parametrize("rng", RANGES)
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("stride", [1, 2])
def test_depthwise(dsq, rng, bits, stride):
    C, shape = 40, (2, 9, 7, 40)
    act = dsq.dsq_quantize_act(torch.rand(shape, device="cuda") * 6, bits, 0.0, 6.0)
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(torch.randn(C, 3, 3, device="cuda") * 0.3, bits, -1.0, 1.0, ws,
                                      depthwise=True, stride=stride, pad=1)
    scale, bias = affine(C, rng)
    both = [dsq.dsq_dwconv2d(act, shape, (bits, 0.0, 6.0), blob, conv, scale, bias, w_offset=0.5,
                             requant=(bits,) + rng, want_f32=f32)[0] for f32 in (True, False)]
    assert torch.equal(*both)
