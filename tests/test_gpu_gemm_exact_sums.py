"""Sums of 1- and 2-bit operands where binary32 accumulators (4-bit floating-point operands) stop
being exact and int8 takes over, large steps of both signs among least ones near 2^23, and
sums of zero."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_gemm_two_pass(2)
    yield d
    d.dsq_set_gemm_two_pass(1)


def codes(gen, lo, hi, *shape):
    return torch.randint(lo, hi, shape, dtype=torch.int8, device="cuda", generator=gen)


@pytest.mark.parametrize("k", [(1 << 23) - 1, 1 << 23, (1 << 23) + 77])   # 4-bit operands; int8
def test_binary(dsq, k):
    gen = torch.Generator(device="cuda").manual_seed(k)
    a, b = codes(gen, 0, 2, 3, k), codes(gen, 0, 2, 5, k)
    a[0], b[0], b[1] = 1, 1, 0                       # the largest sums of both signs
    b[2, : k - k // 32] = 1                          # steps of +-1 far from zero
    C, _ = dsq.dsq_binary_gemm(dsq.dsq_pack_codes(a, 1), dsq.dsq_pack_codes(b, 1), 3, 5, k)
    ref = (2 * a.double() - 1) @ (2 * b.double() - 1).t()
    assert ref[0, 0] == k and ref[0, 1] == -k
    assert torch.equal(C.double(), ref)


def test_2_bit_steps_of_both_signs_near_the_limit(dsq):
    """One accumulator for the whole of K (more tiles than clusters that could split it): -6 a step
    to 95 % of -2^23, then -6, -3, -2, -1, 0, 1 and 3 in random order; the same backwards; and +3 a
    step with -6 among them."""
    m, n, k, few = 1025, 1153, 1398100, 4
    gen = torch.Generator(device="cuda").manual_seed(1)
    head = k - k // 20
    a, b = codes(gen, -2, 2, few, k), codes(gen, 0, 2, few, k) * 2 + 1
    a[:3, :head], b[:3, :head] = -2, 3
    a[1], b[1] = a[0].flip(0), b[0].flip(0)
    a[3], b[3] = 1, 3
    a[3, ::16] = -2
    A, B = (dsq.dsq_pack_codes(t, 2) for t in (a, b))
    ia, ib = torch.arange(m, device="cuda") % few, torch.arange(n, device="cuda") % few
    ws = dsq.new_gemm_workspace(m, n, k, 2)
    C, _ = dsq.dsq_gemm(A[ia].contiguous(), B[ib].contiguous(), m, n, k, 2, ws)
    dsq.check_workspace(ws)
    ref = a.double() @ b.double().t()
    assert ref.min() < -0.94 * 2 ** 23
    assert torch.equal(C.double(), ref[ia][:, ib])


@pytest.mark.parametrize("k", [64, 1000, 7000])
def test_zero_sums_are_positive(dsq, k):
    """Negative codes against zeros: D is the same bit for bit in both forms of dsq_gemm."""
    m, n = 130, 70
    a, b = torch.full((m, k), -2, dtype=torch.int8, device="cuda"), torch.zeros((n, k), dtype=torch.int8, device="cuda")
    a[1::2] = -1
    scale = torch.ones(m, device="cuda")
    scale[::3] = -1.0
    ws = dsq.new_gemm_workspace(m, n, k, 2)
    D = []
    for two in (0, 2):
        dsq.dsq_set_gemm_two_pass(two)
        D.append(dsq.dsq_gemm(dsq.dsq_pack_codes(a, 2), dsq.dsq_pack_codes(b, 2), m, n, k, 2, ws, row_scale=scale)[1])
    dsq.check_workspace(ws)
    assert torch.equal(D[0].view(torch.int32), D[1].view(torch.int32))
    assert torch.equal(torch.signbit(D[1]), (scale < 0)[:, None].expand(m, n))
