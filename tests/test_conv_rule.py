"""The rule by which a dense convolution takes the little-work kernel, against measured times (one
B200, us, back to back in a graph), among them layers that the window kernel refuses (more than
1024 outputs), takes in its plain form or with weights that it expands itself, and
3-bit layers that are left to the im2col kernel."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1908_05033_b200.binding import dsq_conv_t, dsq_nhwc_t, dsq_row_pitch

HERE = os.path.dirname(os.path.abspath(__file__))

# images, side, Cin, Cout, filter, stride, bits, w_offset, fp32 out, little-work kernel, the other one
LAYERS = [
    (4, 7, 512, 1280, 3, 1, 2, 0.5, 0, 8.8, 13.9), (2, 14, 256, 1280, 3, 1, 3, 0.0, 0, 15.5, 19.7),
    (2, 12, 512, 1280, 3, 1, 3, 0.0, 0, 26.1, 30.3), (1, 56, 64, 1280, 3, 2, 3, 0.0, 0, 12.7, 14.3),
    (1, 20, 256, 1280, 3, 1, 3, 0.0, 0, 15.4, 19.8), (2, 28, 128, 1280, 3, 2, 2, 0.5, 0, 6.2, 7.4),
    (4, 30, 64, 1280, 3, 1, 2, 0.0, 0, 31.9, 17.6), (2, 30, 64, 1280, 3, 1, 4, 0.0, 0, 17.3, 8.7),
    (8, 12, 512, 512, 3, 1, 2, 0.0, 0, 12.8, 16.6), (4, 12, 512, 1024, 3, 1, 4, 0.0, 0, 14.4, 17.1),
    (8, 14, 256, 512, 3, 1, 2, 0.0, 0, 12.5, 10.1), (2, 40, 128, 256, 3, 1, 2, 0.0, 0, 10.3, 6.7),
    (4, 20, 256, 512, 3, 1, 2, 0.0, 0, 12.5, 10.0), (2, 20, 256, 256, 3, 1, 4, 0.0, 0, 6.4, 10.4),
    (2, 40, 128, 256, 3, 2, 3, 0.0, 0, 6.8, 9.4), (2, 40, 128, 64, 3, 1, 4, 0.5, 0, 4.8, 6.6),
    (16, 30, 64, 64, 3, 1, 3, 0.5, 0, 12.0, 7.3), (8, 56, 64, 32, 3, 1, 3, 0.5, 0, 11.6, 7.8),
    (8, 56, 16, 16, 3, 1, 3, 0.5, 0, 9.2, 18.1), (8, 28, 96, 96, 3, 1, 3, 0.5, 0, 8.9, 14.9),
    (32, 14, 96, 96, 3, 1, 3, 0.5, 1, 9.2, 13.8), (8, 28, 160, 320, 3, 2, 3, 0.5, 1, 13.0, 18.8),
    (8, 56, 96, 96, 3, 2, 3, 0.5, 0, 8.9, 15.1), (32, 28, 16, 16, 3, 1, 3, 0.5, 1, 9.6, 17.1),
    (32, 14, 128, 256, 1, 1, 3, 0.5, 1, 12.7, 9.6), (32, 7, 160, 64, 3, 2, 3, 0.5, 0, 4.8, 18.2),
    (1, 7, 96, 96, 3, 2, 4, 0.5, 0, 3.4, 8.0), (3, 56, 16, 16, 3, 1, 2, 0.5, 0, 4.8, 6.4),
    (8, 7, 160, 320, 3, 2, 2, 0.5, 0, 3.7, 9.7), (32, 28, 160, 64, 3, 2, 2, 0.5, 0, 7.2, 9.8)]


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("rule") / "conv_rule_host.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", os.path.join(HERE, "conv_rule_host.cpp"), "-o", so],
                   check=True)
    lib = C.CDLL(so)
    lib.window_us.restype = C.c_double
    return lib


def args(n, hw, cin, cout, k, stride):
    return C.byref(dsq_nhwc_t(n, hw, hw, cin)), C.byref(dsq_conv_t(cout, k, k, cin, stride, k // 2, 1))


@pytest.mark.parametrize("n,hw,cin,cout,k,stride,bits,w_offset,f32,small,other", LAYERS)
def test_kernel(rule, n, hw, cin, cout, k, stride, bits, w_offset, f32, small, other):
    shape, conv = args(n, hw, cin, cout, k, stride)
    side = (hw + 2 * (k // 2) - k) // stride + 1
    units = k * k * ((cin + 31) // 32 if bits == 3 else dsq_row_pitch(cin, bits) // 16)
    taken = rule.takes_small(shape, conv, bits, w_offset == 0.5, not f32, n * side * side, (units + 3) // 4)
    assert bool(taken) == (small < other)


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_window_kernel_takes_1024_outputs_at_most(rule, bits):
    for cout, taken in ((1024, True), (1025, False)):
        assert (rule.window_us(*args(2, 14, 256, cout, 3, 1), bits, 1) > 0) == taken


# images, side, Cin, Cout, bits, the window kernel's time with w_offset 0
WINDOW = [
    (1, 40, 128, 32, 2, 6.2), (4, 28, 128, 64, 2, 6.2), (2, 28, 128, 64, 2, 6.1), (8, 12, 512, 32, 2, 13.8),
    (1, 20, 256, 32, 2, 8.6), (4, 7, 512, 32, 2, 13.7), (4, 12, 512, 1024, 2, 16.6), (4, 7, 512, 1024, 2, 16.5),
    (8, 14, 256, 256, 2, 9.9), (32, 7, 512, 512, 2, 16.7)]


@pytest.mark.parametrize("n,hw,cin,cout,bits,us", WINDOW)
def test_window_kernel_without_the_expanded_copy(rule, n, hw, cin, cout, bits, us):
    assert abs(rule.window_us(*args(n, hw, cin, cout, 3, 1), bits, 0) / us - 1) < 0.08


# rows, columns, Cin, Cout, bits, w_offset, the window kernel's time: too wide for windows in one piece
WIDE = [(8, 300, 128, 256, 3, 0.5, 20.2), (4, 520, 64, 64, 4, 0.5, 6.1), (4, 700, 128, 128, 4, 0.5, 9.7),
        (4, 520, 256, 256, 2, 0.0, 16.2), (8, 300, 256, 256, 4, 0.0, 18.4), (4, 520, 64, 128, 3, 0.5, 12.3)]


@pytest.mark.parametrize("h,w,cin,cout,bits,w_offset,us", WIDE)
def test_window_kernel_on_wide_images(rule, h, w, cin, cout, bits, w_offset, us):
    shape, conv = C.byref(dsq_nhwc_t(1, h, w, cin)), C.byref(dsq_conv_t(cout, 3, 3, cin, 1, 1, 1))
    assert abs(rule.window_us(shape, conv, bits, w_offset == 0.5) / us - 1) < 0.15
