"""The little-work GEMM kernel: ragged tiles, rows that end inside a unit, a chunk or a warp's share of
K, odd and even widths, one or both outputs."""
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 1), (1, 31, 33), (16, 32, 128), (17, 33, 127), (15, 30, 129), (33, 65, 255), (40, 100, 31), (200, 136, 300),
         (128, 128, 1023), (64, 64, 4097), (257, 258, 512), (500, 301, 800), (3, 2000, 777), (1200, 7, 64), (18000, 3, 40)]


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("size", SIZES)
def test_little_work(size, bits):
    import paper_1908_05033_b200 as dsq
    m, n, k = size
    g = torch.Generator(device="cuda").manual_seed(m + n + k + bits)
    half = 1 << (bits - 1)
    a = torch.randint(-half, half, (m, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 2 * half, (n, k), dtype=torch.int8, device="cuda", generator=g)
    a[0], b[0] = -half, 2 * half - 1                 # the largest sum
    scale = torch.rand(m, device="cuda", generator=g) - 0.5
    A, B = dsq.dsq_pack_codes(a, bits), dsq.dsq_pack_codes(b, bits)
    ws = dsq.new_gemm_workspace(m, n, k, bits)
    ref = a.double() @ b.double().t()                # whole numbers below 2^53: exact
    torch.cuda.synchronize()
    C, D = dsq.dsq_gemm(A, B, m, n, k, bits, ws, row_scale=scale)
    C1, none = dsq.dsq_gemm(A, B, m, n, k, bits, ws)
    no, D1 = dsq.dsq_gemm(A, B, m, n, k, bits, ws, row_scale=scale, want_i32=False)
    dsq.check_workspace(ws)
    assert none is None and no is None
    assert torch.equal(C.double(), ref) and torch.equal(C1, C)
    assert torch.equal(D, ref.float() * scale[:, None]) and torch.equal(D1, D)
