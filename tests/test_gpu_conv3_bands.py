"""The window kernel's windows of several bands: pairs of image rows (up to 64 output
channels) and stride 2, on odd and even images, tiles that end inside an image, several
planes of channels, one and several passes, every bit width and weight grid."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_conv import conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_conv3_window(3)
    yield d
    d.dsq_set_conv3_window(1)


# N, H, W, Cin, Cout.  Pairs: odd and even heights (a last row alone; the zeros shared with the
# next image), one row, one column, several tiles a CTA, more than 512 positions a band
PAIRS = [(1, 1, 1, 64, 64), (3, 2, 2, 64, 64), (2, 3, 5, 128, 64), (5, 7, 6, 256, 33), (1, 1, 300, 64, 64), (4, 9, 1, 64, 17),
         (2, 57, 57, 64, 64), (3, 56, 56, 64, 40), (1, 6, 255, 128, 64), (1, 5, 700, 64, 64), (1, 40, 40, 512, 64)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("geom", PAIRS)
def test_pairs_of_rows(dsq, geom, bits):
    conv_case(dsq, *geom, 3, 1, 1, bits, 0.5, residual=geom[0] != 3, seed=sum(geom))


# stride 2: even and odd sides, Cout up to 64, one and two planes, one and two window slots
STRIDED = [(1, 1, 1, 64, 64), (2, 2, 2, 128, 128), (3, 3, 3, 64, 65), (2, 5, 4, 256, 128), (1, 8, 9, 512, 200),
           (9, 56, 56, 64, 128), (4, 57, 57, 64, 64), (40, 28, 28, 128, 256), (16, 14, 14, 256, 512), (3, 15, 13, 128, 300),
           (1, 2, 500, 64, 64), (1, 112, 112, 128, 128), (1, 1, 301, 128, 40)]


@pytest.mark.parametrize("w_offset", [0.5, 0.0, 0.3])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("geom", STRIDED)
def test_stride_2(dsq, geom, bits, w_offset):
    conv_case(dsq, *geom, 3, 2, 1, bits, w_offset, residual=geom[0] % 2 == 1, seed=sum(geom))
