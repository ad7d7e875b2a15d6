"""Which form a weight-only GEMM of more than 32 rows takes, against measured times (one B200, us, back to back
in a graph) of problems that the estimates were not fitted to."""
import pytest

from gemm_rules import rules

# M, N, K, the kernel of few rows in blocks of 16 columns, of 32, two passes
FORMS = [(208, 2556, 1600, 24.0, 19.8, 12.5), (271, 2718, 3936, 66.6, 42.6, 21.2), (257, 3016, 656, 18.9, 18.6, 9.3),
         (528, 4676, 672, 55.5, 46.0, 12.6), (1002, 5372, 624, 95.9, 82.5, 15.0), (215, 1852, 5240, 44.0, 31.1, 20.3),
         (56, 812, 1896, 6.5, 8.7, 10.0), (78, 673, 1920, 7.2, 8.5, 9.9), (123, 593, 2128, 7.6, 9.7, 10.7),
         (56, 1287, 1272, 5.6, 7.8, 9.7), (37, 951, 5912, 12.3, 18.8, 18.0), (36, 1956, 656, 3.7, 4.9, 9.2),
         (126, 1613, 1304, 10.0, 8.2, 11.2), (61, 3199, 5848, 29.6, 20.8, 23.8), (41, 4550, 4520, 19.9, 16.1, 26.2),
         (489, 519, 2024, 13.1, 9.6, 10.9), (36, 3017, 2056, 11.2, 8.9, 15.6), (35, 3427, 1120, 8.3, 6.7, 14.3),
         (162, 903, 1208, 7.8, 7.2, 10.5), (148, 1332, 3024, 18.2, 11.9, 13.3)]


@pytest.mark.parametrize("m,n,k,narrow,wide,two", FORMS)
def test_form(rules, m, n, k, narrow, wide, two):
    times = {16: narrow, 32: wide, 0: two}
    assert times[rules.wgemm_form(m, n, k)] <= 1.03 * min(times.values())
