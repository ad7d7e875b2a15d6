"""3-bit operands as 4-bit floating point in the two-pass GEMM: rows that end anywhere inside a chunk
of 32 codes, a packed word or a part of 1024 codes whose sum is kept, and the sums around the limit
up to which binary32 accumulators are exact (int8 beyond)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_gemm_two_pass(2)
    yield d
    d.dsq_set_gemm_two_pass(1)


def check(dsq, a, b):
    (m, k), n = a.shape, b.shape[0]
    ws = dsq.new_gemm_workspace(m, n, k, 3)
    scale = torch.linspace(-1.0, 1.5, m, device="cuda")
    C, D = dsq.dsq_gemm(dsq.dsq_pack_codes(a, 3), dsq.dsq_pack_codes(b, 3), m, n, k, 3, ws, row_scale=scale)
    dsq.check_workspace(ws)
    ref = a.double() @ b.double().t()                # whole numbers below 2^53: exact
    assert torch.equal(C.double(), ref)
    assert torch.equal(D, ref.float() * scale[:, None])
    return ref


@pytest.mark.parametrize("k", [1, 2, 5, 8, 10, 11, 31, 32, 33, 42, 43, 85, 86, 127, 128, 1023, 1024, 1025, 1056, 3000, 8200])
@pytest.mark.parametrize("m,n", [(1, 1), (33, 70), (130, 264)])
def test_row_ends(dsq, m, n, k):
    g = torch.Generator(device="cuda").manual_seed(1000 * k + m)
    a = torch.randint(-4, 4, (m, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 8, (n, k), dtype=torch.int8, device="cuda", generator=g)
    a[0], b[0] = -4, 7                               # the largest sum
    check(dsq, a, b)


@pytest.mark.parametrize("k", [524287, 524288])      # 16 k below 2^23, and not
def test_sums_near_the_limit(dsq, k):
    """Steps of +16 in the accumulator to its limit, then any; the same backwards; -12 a step."""
    g = torch.Generator(device="cuda").manual_seed(k)
    a = torch.randint(-4, 4, (4, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 8, (4, k), dtype=torch.int8, device="cuda", generator=g)
    head = k - k // 20
    a[0], b[0] = -4, 0
    a[1, :head], b[1, :head] = -4, 0
    a[2], b[2] = a[1].flip(0), b[1].flip(0)
    a[3], b[3] = 3, 7
    ref = check(dsq, a, b)
    assert ref[3, 3] == 21 * k and ref[0, 3] == -28 * k
