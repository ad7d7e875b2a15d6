"""dsq_gemm with a workspace of the smallest size and with one that has room for the expanded operands, at
sizes of which the rule says which kernel takes them, and the little-work kernel in each of its blocks, with
rows, columns and K that end inside one: exact results from each."""
import pytest
import torch

from gemm_rules import rules

pytestmark = pytest.mark.gpu

# M, N, K, bits, the form with room and without
FORMS = [(1069, 320, 1732, 3, "two", "small"), (1604, 394, 1027, 3, "two", "small"), (1610, 834, 618, 4, "two", "small"),
         (1500, 1304, 1033, 3, "two", "fused"), (1500, 1303, 1033, 4, "two", "fused"), (200, 136, 300, 2, "small", "small")]


# M, N, K, bits, rows and warps of the little-work kernel's blocks
BLOCKS = [(2159, 93, 15, 2, 16, 4), (53, 148, 5020, 2, 16, 8), (785, 419, 1353, 2, 32, 4), (148, 4467, 820, 2, 32, 4),
          (80, 108, 275, 3, 16, 4), (321, 146, 4002, 3, 16, 8), (2371, 66, 789, 3, 32, 4), (215, 1296, 576, 3, 32, 4),
          (1216, 69, 4136, 3, 32, 8), (25, 3748, 2045, 3, 32, 8), (67, 1554, 349, 4, 16, 4), (25, 538, 2638, 4, 16, 8),
          (1055, 318, 532, 4, 32, 4), (443, 954, 1346, 4, 32, 4), (87, 4507, 197, 4, 32, 4)]


def check(m, n, k, bits):
    import paper_1908_05033_b200 as dsq
    g = torch.Generator(device="cuda").manual_seed(m + n + bits)
    half = 1 << (bits - 1)
    a = torch.randint(-half, half, (m, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 2 * half, (n, k), dtype=torch.int8, device="cuda", generator=g)
    a[-1], b[-1] = -half, 2 * half - 1               # the largest sum
    scale = torch.rand(m, device="cuda", generator=g) - 0.5
    A, B = dsq.dsq_pack_codes(a, bits), dsq.dsq_pack_codes(b, bits)
    ref = a.double() @ b.double().t()                # whole numbers below 2^53: exact
    for ws in (dsq.new_workspace(), dsq.new_gemm_workspace(m, n, k, bits)):
        C, D = dsq.dsq_gemm(A, B, m, n, k, bits, ws, row_scale=scale)
        dsq.check_workspace(ws)
        assert torch.equal(C.double(), ref) and torch.equal(D, ref.float() * scale[:, None])


@pytest.mark.parametrize("m,n,k,bits,with_room,without", FORMS)
def test_form(rules, m, n, k, bits, with_room, without):
    assert rules.gemm_form(m, n, k, bits, 2, True) == with_room and rules.gemm_form(m, n, k, bits, 2, False) == without
    check(m, n, k, bits)


@pytest.mark.parametrize("m,n,k,bits,rows,warps", BLOCKS)
def test_little_work_blocks(rules, m, n, k, bits, rows, warps):
    for outs in (1, 2):
        assert rules.gemm_form(m, n, k, bits, outs, True) == "small"
    assert rules.gemm_small(m, n, k, bits, 2) == (rows, warps)
    check(m, n, k, bits)
