"""Weight-only GEMMs at sizes of which the rules say that each form takes them: two passes with K split
over the pairs of a cluster and rows that are whole sectors or not, one tile, several a pair, and the
kernel of few rows in blocks of 16 and of 32 columns."""
import pytest
import torch

from gemm_rules import rules

pytestmark = pytest.mark.gpu

# columns of a block (0: two passes), parts of K, M, N, K
CASES = [(0, 1, 300, 1000, 64), (0, 1, 9001, 1043, 136), (0, 2, 130, 2304, 2056), (0, 2, 130, 2307, 2056),
         (0, 2, 1000, 1531, 3000), (16, 0, 257, 136, 3072), (16, 0, 40, 2200, 136), (32, 0, 150, 1500, 1000),
         (32, 0, 64, 2395, 136), (32, 0, 64, 4099, 2000)]


@pytest.mark.parametrize("bits", [1, 2, 3, 4])
@pytest.mark.parametrize("columns,split,m,n,k", CASES)
def test_form(rules, columns, split, m, n, k, bits):
    """Small-integer activations: the sums are exact whatever their order."""
    import paper_1908_05033_b200 as dsq
    assert rules.wgemm_form(m, n, k) == columns
    assert columns or rules.tile("bf16", m, n, k)[0][1] == split
    g = torch.Generator(device="cuda").manual_seed(m + n + bits)
    x = torch.randint(-8, 9, (m, k), device="cuda", generator=g).float()
    half = 1 << (bits - 1)
    q = torch.randint(-half, half, (n, k), dtype=torch.int8, device="cuda", generator=g) if bits > 1 else \
        torch.randint(0, 2, (n, k), dtype=torch.int8, device="cuda", generator=g)
    scale = torch.randint(1, 9, (n,), device="cuda", generator=g).float()
    bias = torch.randint(-9, 9, (n,), device="cuda", generator=g).float()
    value = 2 * q.double() + 1 if bits > 1 else 1 - 2 * q.double()     # (a set bit is the signed code -1)
    W, xb = dsq.dsq_pack_codes(q, bits), x.to(torch.bfloat16)
    ref = (x.double() @ value.t()) * scale.double()
    for b in (bias, None):
        y = dsq.dsq_wgemm_bf16(xb, W, m, n, k, bits, scale, b)
        assert torch.equal(y.double(), ref if b is None else ref + b.double())
