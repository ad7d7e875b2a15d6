"""dsq_gemm with a workspace of the smallest size and with one that has room for the expanded operands, at
sizes of which the rule says which kernel takes them: exact results from each."""
import pytest
import torch

from gemm_rules import rules

pytestmark = pytest.mark.gpu

# M, N, K, bits, the form with room and without
FORMS = [(439, 592, 1602, 3, "two", "small"), (1604, 394, 1027, 3, "two", "small"), (1610, 834, 618, 4, "two", "small"),
         (1500, 1304, 1033, 3, "two", "fused"), (1500, 1303, 1033, 4, "two", "fused"), (200, 136, 300, 2, "small", "small")]


@pytest.mark.parametrize("m,n,k,bits,with_room,without", FORMS)
def test_form(rules, m, n, k, bits, with_room, without):
    import paper_1908_05033_b200 as dsq
    assert rules.gemm_form(m, n, k, bits, 2, True) == with_room and rules.gemm_form(m, n, k, bits, 2, False) == without
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
