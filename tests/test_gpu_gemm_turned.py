"""Outputs of the integer GEMMs' second pass that are turned round in shared memory (rows that are not
whole sectors, outputs that are not 32-byte aligned): integers, scaled values and both at once; whole
and ragged tiles, one and several a CTA pair, K whole and split."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# (the last one: whole sectors, but for where the outputs lie)
SIZES = [(1, 31, 64), (129, 33, 100), (300, 257, 1000), (140, 500, 7000), (6000, 1043, 260), (300, 264, 300)]


@pytest.fixture(scope="module")
def dsq():
    import paper_1908_05033_b200 as d
    d.dsq_set_gemm_two_pass(2)
    yield d
    d.dsq_set_gemm_two_pass(1)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("m,n,k", SIZES)
def test_each_output(dsq, m, n, k, bits):
    g = torch.Generator(device="cuda").manual_seed(m + n + bits)
    half = 1 << (bits - 1)
    a = torch.randint(-half, half, (m, k), dtype=torch.int8, device="cuda", generator=g)
    b = torch.randint(0, 2 * half, (n, k), dtype=torch.int8, device="cuda", generator=g)
    a[m // 2] = 0                                    # (+0 times the scale)
    scale = torch.rand(m, device="cuda", generator=g) - 0.5
    A, B = dsq.dsq_pack_codes(a, bits), dsq.dsq_pack_codes(b, bits)
    ws = dsq.new_gemm_workspace(m, n, k, bits)
    ref = a.double() @ b.double().t()                # whole numbers below 2^53: exact
    ref_f = ref.float() * scale[:, None]

    def new(dtype):
        return torch.full((m * n + 4,), 77, dtype=dtype, device="cuda")[4:].view(m, n)    # 16-byte aligned

    for ints, floats in ((True, False), (False, True), (True, True)):
        C, D = new(torch.int32), new(torch.float32)
        dsq.dsq_gemm(A, B, m, n, k, bits, ws, row_scale=scale if floats else None, want_i32=ints,
                     out_i32=C if ints else None, out_f32=D if floats else None)
        dsq.check_workspace(ws)
        assert bool((C == 77).all()) if not ints else torch.equal(C.double(), ref)
        assert bool((D == 77).all()) if not floats else torch.equal(D.view(torch.int32), ref_f.view(torch.int32))
