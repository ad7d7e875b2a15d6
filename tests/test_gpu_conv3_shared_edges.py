"""GPU parity of the window kernel where its loads end around the last image: one row
of zeros is the bottom of an image and the top of the next, and a load that would begin
in the zeros below the last image is written by the kernel instead."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_conv import conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


# N, H, W, Cin, Cout.  Transposed tiles over 20 columns: two loads of 152 positions, the
# second begins 26 .. 5 positions before or behind the image's end (H 5, 6, 7); three
# bands (150 columns or more on plain tiles): the last begins 0 positions behind it
EDGES = [(1, 5, 20, 64, 64), (1, 6, 20, 64, 64), (1, 7, 20, 128, 128), (1, 6, 20, 256, 40), (6, 1, 20, 64, 96),
         (1, 1, 1, 128, 64), (1, 1, 150, 64, 64), (1, 2, 150, 128, 32), (1, 1, 300, 64, 64), (13, 4, 6, 64, 64),
         (5, 17, 1, 64, 64), (1, 3, 224, 64, 64)]


@pytest.mark.parametrize("form", [3, 4])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("geom", EDGES)
def test_shared_edges(dsq, geom, bits, form):
    dsq.dsq_set_conv3_window(form)
    try:
        conv_case(dsq, *geom, 3, 1, 1, bits, 0.5, residual=geom[0] == 1, seed=sum(geom))
    finally:
        dsq.dsq_set_conv3_window(1)
