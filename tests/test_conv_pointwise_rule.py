"""Whether a 1x1 layer from codes to codes, with a residual operand or without, takes the little-work kernel or
the 1x1 kernel, against measured times (one B200, us, back to back in a graph) of layers that the rule was
not fitted to."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1908_05033_b200.binding import dsq_conv_t, dsq_nhwc_t, dsq_row_pitch

HERE = os.path.dirname(os.path.abspath(__file__))

# images, side, Cin, Cout, stride, bits, residual, the little-work kernel's time, the 1x1 kernel's
LAYERS = [
    (5, 20, 960, 512, 1, 2, 0, 8.8, 7.9), (5, 28, 160, 160, 1, 4, 0, 5.8, 4.2), (12, 56, 144, 24, 1, 4, 0, 7.1, 4.9),
    (15, 28, 960, 128, 1, 3, 0, 19.4, 14.1), (5, 28, 144, 160, 1, 3, 0, 7.0, 4.9), (2, 56, 512, 128, 1, 2, 0, 7.6, 5.7),
    (8, 10, 144, 320, 2, 4, 0, 2.6, 3.5), (3, 10, 160, 24, 1, 4, 0, 2.5, 3.4), (2, 33, 96, 16, 2, 2, 0, 2.9, 3.3),
    (9, 14, 512, 256, 1, 3, 0, 5.5, 6.1), (7, 14, 128, 32, 2, 3, 0, 3.0, 3.9), (3, 10, 144, 24, 1, 3, 0, 3.0, 4.1),
    (13, 20, 256, 128, 1, 4, 1, 6.3, 4.8), (10, 28, 960, 128, 1, 3, 1, 14.4, 11.4), (1, 28, 32, 1024, 1, 3, 1, 7.7, 5.5),
    (9, 14, 160, 512, 1, 3, 1, 8.7, 6.2), (10, 28, 160, 128, 1, 2, 1, 7.6, 5.0), (5, 20, 32, 512, 1, 3, 1, 8.2, 5.6),
    (3, 56, 960, 128, 1, 4, 1, 10.5, 8.7), (1, 10, 320, 96, 1, 2, 1, 2.8, 4.4), (2, 20, 96, 512, 1, 3, 1, 4.5, 5.4),
    (1, 20, 96, 128, 1, 4, 1, 2.5, 3.5), (1, 56, 960, 64, 1, 2, 1, 3.8, 6.8), (3, 7, 16, 256, 1, 4, 1, 2.6, 3.4),
    (1, 28, 512, 16, 1, 4, 1, 2.6, 4.7), (5, 7, 144, 24, 1, 3, 1, 3.2, 4.9)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rule") / "conv_pointwise_rule_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", os.path.join(HERE, "conv_pointwise_rule_host.cpp"),
                    "-o", so], check=True)
    return C.CDLL(so)


@pytest.mark.parametrize("n,hw,cin,cout,stride,bits,residual,small,other", LAYERS)
def test_kernel(rule, n, hw, cin, cout, stride, bits, residual, small, other):
    side = (hw - 1) // stride + 1
    units = (cin + 31) // 32 if bits == 3 else dsq_row_pitch(cin, bits) // 16
    taken = rule.takes_small(C.byref(dsq_nhwc_t(n, hw, hw, cin)), C.byref(dsq_conv_t(cout, 1, 1, cin, stride, 0, 1)), bits,
                             n * side * side, (units + 3) // 4, residual)
    assert bool(taken) == (small < other)
