"""Outputs of the weight-only GEMM's second pass: rows that are whole sectors (the last tile of a
CTA turned round in the operand ring, the ones before it not) and rows that are not, one and
several tiles a CTA pair, K whole and split over the pairs of a cluster."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(257, 64, 128), (300, 1000, 64), (9001, 1040, 136), (9001, 1043, 136), (5000, 2504, 64),
                                   (130, 2304, 2056), (257, 136, 3072), (257, 135, 3072)])
@pytest.mark.parametrize("bias", [False, True])
def test_weight_only(m, n, k, bias):
    """Small-integer activations: the sums are exact whatever their order."""
    import paper_1908_05033_b200 as dsq
    g = torch.Generator(device="cuda").manual_seed(m + n)
    x = torch.randint(-8, 9, (m, k), device="cuda", generator=g).float()
    q = torch.randint(-8, 8, (n, k), dtype=torch.int8, device="cuda", generator=g)
    scale = torch.randint(1, 9, (n,), device="cuda", generator=g).float()
    b = torch.randint(-9, 9, (n,), device="cuda", generator=g).float()
    ws = torch.zeros(dsq.lib.dsq_wgemm_workspace_bytes(n, k), dtype=torch.uint8, device="cuda")
    y = dsq.dsq_wgemm_bf16(x.to(torch.bfloat16), dsq.dsq_pack_codes(q, 4), m, n, k, 4, scale, b if bias else None, ws=ws)
    dsq.check_workspace(ws)
    ref = (x.double() @ (2 * q.double() + 1).t()) * scale.double()
    assert torch.equal(y.double(), ref + b.double() if bias else ref)
