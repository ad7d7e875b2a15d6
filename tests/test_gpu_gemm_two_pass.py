"""GPU parity of the two-pass GEMMs where K is split over a cluster's pairs and at
widths that are not a multiple of a store."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from oracle import binary, native
import dsq_inputs
from gpu_util import T, N


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    return d


# one tile and many, K of 12 to 50 blocks of 128 (split from 24 on), odd, even and
# multiple-of-8 widths
SIZES = [(1, 1, 3072), (256, 256, 3073), (300, 257, 3100), (513, 130, 6400), (700, 1028, 3200),
         (260, 1026, 1700), (2100, 515, 3080), (130, 2304, 3333)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("size", SIZES)
def test_two_pass_gemm(dsq, size, bits):
    M, Nn, K = size
    A, B, rs = dsq_inputs.gemm_case(M, Nn, K, bits)
    dsq.dsq_set_gemm_two_pass(2)
    try:
        ws = dsq.new_gemm_workspace(M, Nn, K, bits)
        Cg, Dg = dsq.dsq_gemm(dsq.dsq_pack_codes(T(A), bits), dsq.dsq_pack_codes(T(B), bits), M, Nn,
                              K, bits, ws, row_scale=T(rs))
        dsq.check_workspace(ws)
    finally:
        dsq.dsq_set_gemm_two_pass(1)
    C = native.gemm(A, B)
    assert np.array_equal(N(Cg), C)
    assert np.array_equal(N(Dg), native.gemm_dequant(C, rs))


@pytest.mark.parametrize("size", SIZES)
def test_binary_gemm(dsq, size):
    M, Nn, K = size
    A, B, _ = dsq_inputs.binary_gemm_case(M, Nn, K)
    Cg, _ = dsq.dsq_binary_gemm(dsq.dsq_pack_codes(T(A), 1), dsq.dsq_pack_codes(T(B), 1), M, Nn, K)
    assert np.array_equal(N(Cg), binary.binary_gemm(A, B))


@pytest.mark.parametrize("size", [(257, 300, 1536), (600, 1028, 1600), (130, 2051, 2056)])
def test_weight_only_gemm_split(dsq, size):
    """Small-integer activations: sums are exact whatever their order."""
    M, Nn, K = size
    rng = np.random.default_rng(3)
    x = rng.integers(-8, 9, (M, K)).astype(np.float32)
    q = rng.integers(0, 16, (Nn, K)).astype(np.int16)
    Wp = dsq.dsq_pack_codes(T((q - 8).astype(np.int8)), 4)
    Y = dsq.dsq_wgemm_bf16(T(x).to(torch.bfloat16), Wp, M, Nn, K, 4, T(np.ones(Nn, np.float32)), None)
    want = x.astype(np.int64) @ (2 * (q.astype(np.int64) - 8) + 1).T
    assert np.array_equal(N(Y).astype(np.int64), want)
