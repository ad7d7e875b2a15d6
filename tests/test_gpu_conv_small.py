"""GPU parity of the kernel for convolutions with little work at the edges of its
tiles, and of the larger layers' kernels on the same small problems."""
import pytest

pytestmark = pytest.mark.gpu

from test_gpu_conv import GEOMS, conv_case


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


# N, H, W, Cin, Cout, k, stride, pad: single pixels, ragged pixel and channel tiles,
# units past a pixel's row (3-bit), K of one unit and of many chunks
EDGES = [(1, 1, 1, 1, 1, 1, 1, 0), (1, 1, 1, 33, 65, 3, 1, 1), (1, 3, 5, 40, 31, 3, 2, 1),
         (3, 4, 4, 96, 33, 1, 1, 0), (1, 7, 7, 512, 512, 3, 1, 1), (2, 5, 3, 1000, 24, 1, 2, 0),
         (1, 17, 15, 66, 129, 3, 1, 0), (4, 9, 9, 130, 40, 3, 1, 1), (1, 56, 56, 24, 144, 1, 1, 0)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("geom", EDGES)
def test_small_conv(dsq, geom, residual, bits):
    conv_case(dsq, *geom, bits, 0.5, residual=residual, seed=sum(geom), out_rng=(-0.5, 1.0))


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("geom", GEOMS)
def test_other_kernels_on_small_problems(dsq, geom, bits):
    dsq.dsq_set_conv3_window(3)          # (a set hook leaves the small kernel out)
    try:
        conv_case(dsq, *geom, bits, 0.5, residual=True, seed=sum(geom))
    finally:
        dsq.dsq_set_conv3_window(1)
