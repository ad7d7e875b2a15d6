"""The window kernel's 2-bit form on 4-bit floating-point operands: sizes around its tiles of
240 positions, its three row lengths (64, 128, 256 and more channels), windows in one piece
and in three bands, the largest sums, and a blob whose expanded copy is not of that form."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from oracle import native
from gpu_util import T, N
from test_gpu_conv import conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_conv3_window(3)
    yield d
    d.dsq_set_conv3_window(1)


# N, H, W, Cin, Cout: 239, 240 and 241 positions up to the last pixel; several tiles a CTA;
# 250 and 251 columns (the last in one piece, the first in bands) with one and two slots
GEOMS = [(1, 1, 239, 64, 64), (1, 1, 240, 128, 128), (1, 1, 241, 256, 40), (1, 16, 14, 64, 65), (1, 15, 15, 512, 130),
         (9, 56, 56, 64, 64), (5, 60, 60, 128, 200), (1, 3, 250, 64, 33), (1, 3, 251, 64, 64), (2, 2, 251, 128, 128),
         (1, 4, 250, 256, 100), (1, 4, 300, 256, 256), (1, 3, 600, 1024, 24)]


@pytest.mark.parametrize("geom", GEOMS)
def test_shapes(dsq, geom):
    conv_case(dsq, *geom, 3, 1, 1, 2, 0.5, residual=geom[0] % 2 == 1, seed=sum(geom))


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("geom", [(149, 10, 10, 64, 64), (70, 12, 13, 128, 128), (37, 13, 12, 256, 256), (64, 7, 7, 512, 512),
                                  (90, 14, 14, 128, 40)])
def test_tiles_of_fewer_positions(dsq, geom, bits):
    """One pass of 112 .. 240 positions a tile (columns of a tile that the warps of a
    tensor-memory quarter share unevenly) and two passes."""
    conv_case(dsq, *geom, 3, 1, 1, bits, 0.5, residual=geom[3] != 128, seed=sum(geom))


@pytest.mark.parametrize("cin", [64, 128, 256, 1024])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_largest_sums(dsq, cin, sign):
    """Every product 3 * (+-3), and one weight of a channel that differs by the least step:
    the sums are whole numbers up to 9 * 9 * 1024 and exact."""
    h, w, co = 9, 31, 72
    x = np.full((1, h, w, cin), 2.0, np.float32)
    wt = np.full((co, 3, 3, cin), 0.1 * sign, np.float32)
    wt[np.arange(co), 1, 1, np.arange(co) % cin] = 0.03 * sign
    acc, sa = native.conv2d(native.quantize(x, 2, 0.0, 2.0), native.quantize_weights(wt, 2, -0.1, 0.1), 1, 1,
                            want_sa=True)
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(T(wt), 2, -0.1, 0.1, ws, stride=1, pad=1)
    one = torch.ones(co, device="cuda")
    _, y, got = dsq.dsq_conv2d(dsq.dsq_quantize_act(T(x), 2, 0.0, 2.0), x.shape, (2, 0.0, 2.0), blob, conv, one,
                               0 * one, ws, w_offset=0.5, want_f32=True, want_acc=True)
    assert dsq.dsq_workspace_status(ws) == 0
    assert np.array_equal(N(got), 2 * acc + sa[..., None])
    assert np.array_equal(N(y), (2 * acc + sa[..., None]).astype(np.float32) * np.float32(0.5))


def test_unmarked_copy_is_refused(dsq):
    """A blob kept from a library that stored the copy as int8: an error, not wrong sums."""
    ws = dsq.new_workspace()
    blob, conv = dsq.dsq_pack_weights(torch.randn(64, 3, 3, 128, device="cuda") * 0.05, 2, -0.1, 0.1, ws, stride=1,
                                      pad=1)
    act = dsq.dsq_quantize_act(torch.rand(2, 20, 20, 128, device="cuda"), 2, 0.0, 2.0)
    one = torch.ones(64, device="cuda")
    args = (act, (2, 20, 20, 128), (2, 0.0, 2.0), blob, conv, one, one, ws)
    dsq.dsq_conv2d(*args, w_offset=0.5, requant=(2, 0.0, 2.0))
    assert dsq.dsq_workspace_status(ws) == 0
    kept = blob[-16:].clone()
    blob[-16:] = 0x41
    dsq.dsq_conv2d(*args, w_offset=0.5, requant=(2, 0.0, 2.0))
    assert dsq.dsq_workspace_status(ws) == -8, "DSQ_ERR_UNSUPPORTED"
    blob[-16:] = kept
    dsq.dsq_conv2d(*args, w_offset=0.5, requant=(2, 0.0, 2.0))
    assert dsq.dsq_workspace_status(ws) == 0
