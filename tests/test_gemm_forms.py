"""Which of its kernels dsq_gemm takes, against measured times (one B200, us, back to back in a graph)."""
import pytest

from gemm_rules import rules

# M, N, K, bits, arrays written, the fused kernel's time, two passes', the little-work kernel's
FORMS = [(1069, 320, 1732, 3, 2, 12.7, 8.9, 9.9), (439, 592, 1602, 3, 2, 13.4, 8.6, 7.9), (1604, 394, 1027, 3, 1, 14.1, 8.2, 11.9),
         (181, 2160, 1737, 3, 2, 13.8, 8.8, 11.1), (1610, 834, 618, 4, 1, 15.5, 8.5, 10.0), (291, 1086, 1962, 3, 1, 15.9, 8.2, 9.8)]


@pytest.mark.parametrize("m,n,k,bits,outs,fused,two,small", FORMS)
def test_without_room_for_two_passes(rules, m, n, k, bits, outs, fused, two, small):
    """A workspace of the smallest size leaves the fused kernel and the little-work one."""
    assert rules.gemm_form(m, n, k, bits, outs, False) == "small" and small < fused
