"""GPU parity of the weight-only GEMM for few rows at the edges of its tiles."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

import dsq_inputs
from oracle import weight_only
from test_gpu_binary_weight_only import run_wgemm


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("size", [(1, 33, 8), (15, 17, 120), (16, 40, 136), (17, 31, 1032),
                                  (33, 70, 264), (64, 65, 2056), (65, 33, 128), (3, 3600, 392),
                                  (31, 4100, 160), (5, 2368, 136), (20, 2369, 136)])
def test_few_rows(dsq, size, bits):
    M, Nn, K = size
    x, q, u, bias = dsq_inputs.weight_only_case(M, Nn, K, bits)
    for w_offset in (0.5, 0.0):
        Yg, scale = run_wgemm(dsq, x, q, u, bias, bits, w_offset)
        s = scale.astype(np.float64)
        if w_offset == 0.5:
            u_eff = s * (2 ** bits - 1)
            Y = weight_only.linear(x, q, bits, -u_eff, u_eff, bias)
            mag = weight_only.abs_linear(x, q, bits, -u_eff, u_eff)
        else:
            c = q.astype(np.float64) - (1 << (bits - 1))
            Y = (x.astype(np.float64) @ c.T) * s + bias
            mag = (np.abs(x.astype(np.float64)) @ np.abs(c).T) * s
        tol = K * 2.0 ** -23 * mag + 1e-6 * np.abs(Y) + 1e-30
        assert np.all(np.abs(Yg - Y) <= tol)
