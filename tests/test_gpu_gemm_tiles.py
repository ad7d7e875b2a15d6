"""The second pass of the two-pass GEMMs over its tile widths (64 to 256 columns, the last tile
of a row ragged), one and several tiles a CTA pair, rows of outputs that are whole sectors
or not, and the 4-bit floating-point operands of 1 and 2 bits up to their largest sums."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from oracle import native
from gpu_util import T, N


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_gemm_two_pass(2)
    yield d
    d.dsq_set_gemm_two_pass(1)


SIZES = [(300, 64, 700), (257, 95, 256), (129, 33, 255), (2500, 1111, 500), (3136, 512, 700), (5000, 2000, 300),
         (19000, 250, 260), (700, 6001, 513), (4000, 3001, 257), (520, 450, 7000)]


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("size", SIZES)
def test_integer(dsq, size, bits):
    m, n, k = size
    g = torch.Generator(device="cuda").manual_seed(m + n + k + bits)
    half = 1 << (bits - 1)
    a = torch.randint(-half, half, (m, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 2 * half, (n, k), dtype=torch.int8, device="cuda", generator=g)
    scale = torch.rand(m, device="cuda", generator=g) + 0.5
    if bits == 1:
        a, b = a & 1, b & 1
        A, B = 2 * a.double() - 1, 2 * b.double() - 1
        C, D = dsq.dsq_binary_gemm(dsq.dsq_pack_codes(a, 1), dsq.dsq_pack_codes(b, 1), m, n, k, row_scale=scale)
    else:
        A, B = a.double(), b.double()
        ws = dsq.new_gemm_workspace(m, n, k, bits)
        C, D = dsq.dsq_gemm(dsq.dsq_pack_codes(a, bits), dsq.dsq_pack_codes(b, bits), m, n, k, bits, ws,
                            row_scale=scale)
        dsq.check_workspace(ws)
    ref = A @ B.t()                                  # whole numbers below 2^53: exact
    assert torch.equal(C.double(), ref)
    assert torch.equal(D, ref.float() * scale[:, None])


@pytest.mark.parametrize("k", [1398100, 1398103])    # 6 k below 2^23: 4-bit operands; not: int8
@pytest.mark.parametrize("b_last", [3, 2])
def test_largest_2_bit_sums(dsq, k, b_last):
    a, b = np.full((1, k), -2, np.int8), np.full((2, k), 3, np.int8)
    b[1, -1] = b_last
    b[1, : k // 2] = 1
    ws = dsq.new_gemm_workspace(1, 2, k, 2)
    C, _ = dsq.dsq_gemm(dsq.dsq_pack_codes(T(a), 2), dsq.dsq_pack_codes(T(b), 2), 1, 2, k, 2, ws)
    dsq.check_workspace(ws)
    assert np.array_equal(N(C), native.gemm(a, b))


@pytest.mark.parametrize("size", [(300, 64, 704), (257, 95, 256), (2500, 1111, 504), (700, 6001, 520), (520, 452, 3504)])
def test_weight_only(dsq, size):
    """Small-integer activations: the sums are exact whatever their order."""
    m, n, k = size
    g = torch.Generator(device="cuda").manual_seed(m + n)
    x = torch.randint(-8, 9, (m, k), device="cuda", generator=g).float()
    q = torch.randint(-4, 4, (n, k), dtype=torch.int8, device="cuda", generator=g)
    bias = torch.randint(-9, 9, (n,), device="cuda", generator=g).float()
    y = dsq.dsq_wgemm_bf16(x.to(torch.bfloat16), dsq.dsq_pack_codes(q, 3), m, n, k, 3, torch.full((n,), 2.0, device="cuda"),
                           bias)
    # (col_scale is half of the grid's step: 2 c + 1)
    ref = x.double() @ (2 * q.double() + 1).t()
    assert torch.equal(y.double(), 2 * ref + bias.double())
