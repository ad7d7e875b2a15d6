"""GPU parity of the window kernel's transposed tiles on 3-bit codes: the rows' words
are put together from 24-bit pieces, so output channels around every multiple of 8, 32
and 128 and rows with spare words behind the codes."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_conv import conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


# N, H, W, Cin, Cout: 64 channels take two filter taps a K step, wider ones planes of 128
EDGES = [(1, 9, 11, 64, 1), (2, 17, 13, 64, 40), (1, 16, 31, 64, 43), (1, 5, 7, 64, 64), (2, 9, 21, 64, 65),
         (1, 15, 15, 128, 64), (1, 12, 10, 128, 96), (1, 6, 6, 256, 131), (1, 3, 250, 64, 32)]


@pytest.mark.parametrize("rng,w_offset", [((0.0, 1.0), 0.5), ((-0.5, 1.0), 0.5), ((0.0, 1.0), 0.25)])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("geom", EDGES)
def test_transposed_3bit(dsq, geom, residual, rng, w_offset):
    dsq.dsq_set_conv3_window(3)          # (a set hook leaves the small kernel out)
    try:
        conv_case(dsq, *geom, 3, 1, 1, 3, w_offset, residual=residual, seed=sum(geom), out_rng=rng)
    finally:
        dsq.dsq_set_conv3_window(1)
