"""The weight-only GEMM of few rows in blocks of 64 rows x 32 columns: ragged rows, columns and
shares of K."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("m,n,k", [(150, 1500, 1000), (64, 2395, 136), (33, 2400, 1032), (100, 2371, 520), (300, 790, 776)])
def test_wide_blocks(m, n, k, bits):
    """Small-integer activations: the sums are exact whatever their order."""
    import paper_1908_05033_b200 as dsq
    g = torch.Generator(device="cuda").manual_seed(m + n)
    x = torch.randint(-8, 9, (m, k), device="cuda", generator=g).float()
    half = 1 << (bits - 1)
    q = torch.randint(-half, half, (n, k), dtype=torch.int8, device="cuda", generator=g) if bits > 1 else \
        torch.randint(0, 2, (n, k), dtype=torch.int8, device="cuda", generator=g)
    scale = torch.randint(1, 9, (n,), device="cuda", generator=g).float()
    bias = torch.randint(-9, 9, (n,), device="cuda", generator=g).float()
    value = 2 * q.double() + 1 if bits > 1 else 1 - 2 * q.double()     # (a set bit is the signed code -1)
    y = dsq.dsq_wgemm_bf16(x.to(torch.bfloat16), dsq.dsq_pack_codes(q, bits), m, n, k, bits, scale, bias)
    assert torch.equal(y.double(), (x.double() @ value.t()) * scale.double() + bias.double())
