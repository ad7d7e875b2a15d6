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


# M, N, K, bits, arrays written, the faster of the other kernels, the little-work kernel in blocks of 16
# rows and 4, 16 and 8, 32 and 4, 32 rows and 8 warps (problems that its estimate was not fitted to)
BLOCKS = [(267, 16, 234, 2, 2, 4.6, 1.9, 2.0, 2.7, 2.3), (410, 624, 19, 2, 1, 4.3, 2.3, 3.8, 3.3, 4.1),
          (989, 147, 469, 3, 2, 8.2, 3.4, 5.5, 4.0, 4.7), (718, 81, 114, 3, 1, 5.5, 2.0, 2.1, 2.8, 2.5),
          (4200, 605, 25, 4, 1, 21.6, 12.7, 24.1, 13.2, 26.8), (1031, 28, 276, 4, 1, 5.2, 1.6, 1.8, 1.9, 1.8),
          (320, 176, 3982, 2, 2, 10.7, 3.3, 3.1, 4.7, 4.0), (37, 1467, 5575, 2, 1, 14.5, 3.9, 3.7, 5.6, 5.1),
          (24, 40, 6112, 4, 1, 15.1, 4.6, 3.7, 5.6, 4.8), (173, 32, 5148, 4, 2, 14.2, 4.5, 3.8, 5.7, 4.8),
          (2412, 136, 44, 2, 2, 3.8, 3.6, 5.3, 3.2, 6.0), (385, 976, 1487, 2, 1, 6.9, 5.0, 6.7, 4.3, 6.8),
          (4263, 64, 3203, 3, 1, 19.8, 12.2, 16.5, 10.2, 11.3), (64, 4400, 409, 3, 2, 6.2, 4.9, 7.7, 3.9, 5.0),
          (1778, 394, 1547, 3, 1, 9.2, 15.6, 26.7, 14.9, 17.9), (139, 2430, 992, 4, 1, 7.5, 4.4, 5.2, 3.6, 5.8),
          (700, 584, 3181, 4, 1, 10.0, 7.9, 9.4, 6.7, 9.1), (3744, 16, 3765, 3, 1, 22.9, 10.7, 9.3, 7.5, 6.8),
          (19, 3082, 4585, 3, 2, 25.7, 9.0, 10.3, 8.0, 7.6)]


@pytest.mark.parametrize("m,n,k,bits,outs,other,a,b,c,d", BLOCKS)
def test_little_work_blocks(rules, m, n, k, bits, outs, other, a, b, c, d):
    times = {(16, 4): a, (16, 8): b, (32, 4): c, (32, 8): d}
    taken = rules.gemm_form(m, n, k, bits, outs, True)
    assert (taken == "small") == (min(times.values()) < other)
    assert times[rules.gemm_small(m, n, k, bits, outs)] <= 1.04 * min(times.values())


# M, N, K, the fused kernel's time, two passes' (operands as 4-bit floating point): 3-bit codes
PASSES = [(2558, 248, 210, 6.3, 6.7), (3015, 1420, 184, 9.7, 11.8), (427, 1516, 265, 6.4, 7.1), (625, 2288, 147, 6.8, 7.7),
          (4505, 140, 381, 6.0, 7.8), (1039, 848, 322, 6.4, 7.3), (188, 356, 284, 5.4, 7.8), (254, 336, 1271, 10.1, 6.9),
          (193, 735, 1316, 13.9, 8.7), (145, 1377, 2038, 15.5, 7.8), (473, 273, 505, 7.1, 6.5), (2982, 136, 1471, 11.8, 8.9),
          (2400, 1114, 2702, 57.7, 17.5), (2286, 428, 3731, 23.9, 12.6), (2497, 1287, 171, 42.7, 15.4)]


@pytest.mark.parametrize("m,n,k,fused,two", PASSES)
def test_three_bits_in_two_passes(rules, m, n, k, fused, two):
    _, clocks = rules.tile("f4", m, n, k)
    assert bool(rules.two_passes(m, n, k, 3, True, clocks)) == (two < fused)
