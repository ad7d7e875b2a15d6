"""The little-work convolution kernel where a warp walks several chunks of K and asks for the next
one's words ahead: one to nine chunks a warp, the last of them whole, partial or past the end of
the filter, in tiles of one and of two pixel rows, at image corners."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_conv import conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


# images, side, Cin, Cout, filter, stride: 5 to 36 chunks (3 bits: up to 72) over 4 to 16 warps
LAYERS = [(1, 5, 64, 32, 3, 1), (1, 9, 96, 40, 3, 2), (1, 14, 256, 64, 3, 1), (1, 7, 512, 256, 3, 1), (2, 7, 512, 512, 3, 2),
          (8, 7, 512, 512, 3, 1), (6, 11, 272, 128, 3, 1), (3, 14, 960, 160, 1, 1), (5, 13, 200, 96, 3, 1)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("layer", LAYERS)
def test_chunks_ahead(dsq, layer, bits):
    n, hw, ci, co, k, s = layer
    conv_case(dsq, n, hw, hw, ci, co, k, s, k // 2, bits, 0.5, residual=co % 64 == 0)
