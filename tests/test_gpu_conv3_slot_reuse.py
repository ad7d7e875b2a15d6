"""The window kernel where a CTA works on two windows and its weights come through the
packed ring, on images wide enough that the ring's warps wait long for an operand stage: a
slot of the ring is filled again only after every warp has read it.  Repeated launches
against the im2col kernel (both are compared with the oracle elsewhere)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# bits, N, H, W, Cin, Cout, w_offset: two tiles a CTA (one and three bands a window), two planes
CASES = [(3, 6, 14, 224, 128, 128, 0.5), (3, 2, 37, 257, 128, 128, 0.0), (3, 11, 13, 141, 64, 139, 0.5),
         (3, 8, 15, 224, 64, 128, 0.3), (4, 3, 23, 150, 256, 81, 0.3), (2, 8, 15, 224, 128, 100, 0.0)]


@pytest.mark.parametrize("form", [3, 4])
@pytest.mark.parametrize("case", CASES)
def test_slot_reuse(case, form):
    import paper_1908_05033_b200 as dsq
    bits, n, h, w, ci, co, w_offset = case
    torch.manual_seed(bits + h)
    ws = dsq.new_workspace()
    act = dsq.dsq_quantize_act(torch.rand(n, h, w, ci, device="cuda") * 2, bits, 0.0, 2.0)
    blob, conv = dsq.dsq_pack_weights(torch.randn(co, 3, 3, ci, device="cuda") * 0.05, bits, -0.1, 0.1, ws,
                                      stride=1, pad=1)
    scale = torch.full((co,), 0.01, device="cuda")
    bias = torch.randn(co, device="cuda")

    def run(hook, **kw):
        dsq.dsq_set_conv3_window(hook)
        try:
            return dsq.dsq_conv2d(act, (n, h, w, ci), (bits, 0.0, 2.0), blob, conv, scale, bias, ws,
                                  w_offset=w_offset, requant=(bits, 0.0, 3.0), **kw)
        finally:
            dsq.dsq_set_conv3_window(1)

    codes, _, acc = run(0, want_acc=True)
    for _ in range(8):
        c, _, a = run(form, want_acc=True)
        assert torch.equal(a, acc) and torch.equal(c, codes)
        assert torch.equal(run(form)[0], codes)
    assert dsq.dsq_workspace_status(ws) == 0
