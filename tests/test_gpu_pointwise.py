"""GPU parity of the 1x1 convolution kernel (codes to codes) at the edges of its
tiles, and of the lean codes epilogue on channels that are not finite."""
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
    return d


# N, H, W, Cin, Cout, stride
GEOMS = [(1, 1, 1, 3, 5, 1), (1, 5, 5, 16, 96, 1), (2, 8, 8, 129, 33, 1), (1, 11, 13, 144, 300, 1),
         (1, 9, 9, 960, 320, 1), (3, 7, 7, 320, 1280, 1), (2, 15, 15, 64, 130, 2),
         (3, 14, 14, 256, 512, 2), (1, 1, 1, 40, 8, 2),
         # many tiles per CTA: 512- and 256-pixel tiles, a ragged last one
         (5, 151, 149, 16, 16, 1), (3, 131, 131, 24, 144, 1), (9, 120, 120, 64, 32, 2)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("residual", [False, True])
@pytest.mark.parametrize("geom", GEOMS)
def test_pointwise(dsq, geom, residual, bits):
    n, h, w, ci, co, s = geom
    conv_case(dsq, n, h, w, ci, co, 1, s, 0, bits, 0.5, residual=residual, seed=ci + co,
              out_rng=(-0.7, 1.3) if s == 2 else (0.0, 1.0))
    if (n, h) == (1, 5):
        conv_case(dsq, n, h, w, ci, co, 1, s, 0, bits, 0.0, residual=residual, per_channel=True)


@pytest.mark.parametrize("depthwise", [False, True])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_channels_that_are_not_finite(dsq, bits, depthwise):
    """NaN and infinite scales and biases, and scales at the ends of the range:
    the codes of the pinned sequence (NaN -> code 0)."""
    rng = np.random.default_rng(3)
    inf, nan = np.inf, np.nan
    vals = [nan, inf, -inf, 0.0, 0.02, -0.02, 1e29, -1e29, 1e-30]
    scale = np.array([a for a in vals for _ in vals], np.float32)
    bias = np.array([b for _ in vals for b in vals], np.float32)
    C = scale.size
    q = rng.integers(0, 2 ** bits, (2, 6, 5, C), dtype=np.int8)
    q[0, 0, :2] = 0                                      # accumulators of exactly 0
    if depthwise:
        w = rng.standard_normal((C, 3, 3)).astype(np.float32)
        cw = native.quantize_weights(w.reshape(C, 9), bits, -1.0, 1.0).reshape(C, 3, 3)
        acc = native.dwconv2d(q, cw, 1, 1)
    else:
        w = rng.standard_normal((C, 1, 1, C)).astype(np.float32)
        cw = native.quantize_weights(w, bits, -1.0, 1.0)
        acc = native.conv2d(q, cw, 1, 0)
    with np.errstate(all="ignore"):
        y = native.epilogue(acc, scale, bias)
    want = native.pack_rows(native.quantize(y, bits, 0.0, 2.0).reshape(-1, C), bits)
    ws = dsq.new_workspace()
    act = T(native.pack_rows(q.reshape(-1, C), bits)).view(2, 6, 5, -1)
    blob, conv = dsq.dsq_pack_weights(T(w), bits, -1.0, 1.0, ws, depthwise=depthwise, stride=1,
                                      pad=1 if depthwise else 0)
    args = (act, q.shape, (bits, 0.0, 2.0), blob, conv, T(scale), T(bias))
    codes, _, _ = dsq.dsq_dwconv2d(*args, requant=(bits, 0.0, 2.0)) if depthwise else \
        dsq.dsq_conv2d(*args, ws, requant=(bits, 0.0, 2.0))
    assert np.array_equal(N(codes).reshape(want.shape), want)
