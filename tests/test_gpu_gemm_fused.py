"""The fused GEMM kernel (both operands expanded tile by tile) on sizes that are otherwise left to the
little-work kernel or the two passes: remainders of rows, columns and K, rows of outputs of any
width, the largest sums, and a call right after one whose wait ran out."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from oracle import native
import dsq_inputs
from gpu_util import T, N


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_gemm_two_pass(0)
    yield d
    d.dsq_set_gemm_two_pass(1)


def run(dsq, A, B, rs, bits):
    m, k = A.shape
    ws = dsq.new_workspace()
    got = dsq.dsq_gemm(dsq.dsq_pack_codes(T(A), bits), dsq.dsq_pack_codes(T(B), bits), m, B.shape[0], k, bits, ws,
                       row_scale=T(rs))
    assert dsq.dsq_workspace_status(ws) == 0
    return N(got[0]), N(got[1])


SIZES = [(1, 1, 1), (128, 32, 128), (128, 256, 128), (130, 70, 200), (300, 257, 1000), (129, 513, 129), (64, 48, 4096),
         (515, 130, 771), (130, 72, 200), (300, 260, 1000), (257, 516, 300), (18000, 3, 40), (700, 1030, 1100)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("size", SIZES)
def test_ragged(dsq, bits, size):
    A, B, rs = dsq_inputs.gemm_case(*size, bits)
    ref = native.gemm(A, B)
    Cg, Dg = run(dsq, A, B, rs, bits)
    assert np.array_equal(ref, Cg)
    assert np.array_equal(native.gemm_dequant(ref, rs), Dg)


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_extreme_codes(dsq, bits):
    half = 1 << (bits - 1)
    m, n, k = 128, 64, 8192
    B = np.full((n, k), 2 * half - 1, np.int8)
    for code in (-half, half - 1, 0):
        Cg, Dg = run(dsq, np.full((m, k), code, np.int8), B, np.ones(m, np.float32), bits)
        assert np.all(Cg == k * code * (2 * half - 1)) and np.all(Dg == Cg)


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_call_after_a_wait_that_ran_out(dsq, bits):
    """The producer of the packed rows leaves out one round: the kernel returns with the status of
    a timeout, and the same kernel launched right after gives the oracle's result."""
    m, n, k = 128, 64, 1024
    A, B, rs = dsq_inputs.gemm_case(m, n, k, bits)
    ref = native.gemm(A, B)
    ws = dsq.new_workspace()
    Ap, Bp = dsq.dsq_pack_codes(T(A), bits), dsq.dsq_pack_codes(T(B), bits)
    for skip in (0, 2):
        dsq.dsq_set_wait_limit_ns(3_000_000)
        dsq.dsq_set_test_skip_b_round(skip)
        try:
            dsq.dsq_gemm(Ap, Bp, m, n, k, bits, ws)
            torch.cuda.synchronize()
        finally:
            dsq.dsq_set_test_skip_b_round(-1)
            dsq.dsq_set_wait_limit_ns(0)
        assert dsq.dsq_workspace_status(ws) == -10          # DSQ_ERR_TIMEOUT
        Cg, Dg = dsq.dsq_gemm(Ap, Bp, m, n, k, bits, ws, row_scale=T(rs))
        assert dsq.dsq_workspace_status(ws) == 0
        assert np.array_equal(N(Cg), ref)
        assert np.array_equal(N(Dg), native.gemm_dequant(ref, rs))


def test_static_workspace(dsq):
    """Calls that meet each other's leftovers in the static scratch."""
    stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
    for m, n, k, bits in [(300, 257, 1000, 4), (515, 130, 771, 2), (129, 66, 1000, 3)] * 2:
        A, B, rs = dsq_inputs.gemm_case(m, n, k, bits)
        Ap, Bp, rs_t = dsq.dsq_pack_codes(T(A), bits), dsq.dsq_pack_codes(T(B), bits), T(rs)
        Cg = torch.full((m, n), -1, dtype=torch.int32, device="cuda")
        Dg = torch.full((m, n), float("nan"), device="cuda")
        st = dsq.lib.dsq_gemm_static_ws(*(C.c_void_p(t.data_ptr()) for t in (Ap, Bp)), m, n, k, bits,
                                        *(C.c_void_p(t.data_ptr()) for t in (Cg, rs_t, Dg)), 1, stream)
        assert st == 0
        ref = native.gemm(A, B)
        assert np.array_equal(N(Cg), ref)
        assert np.array_equal(N(Dg), native.gemm_dequant(ref, rs))
