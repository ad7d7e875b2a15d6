"""Inside a recorded pass the kernels read weights, scales and biases before the kernel
ahead of them has completed: rewritten in place between two passes, on the same stream and
with nothing waited for, the new ones are used by every layer, the first included."""
import pytest
import torch

pytestmark = pytest.mark.gpu

import dsq_inputs
from dsq_inputs import Layer
from gpu_util import T


def wide_stack(bits):
    """Enough work that the window, 1x1, depthwise and im2col kernels take their layers."""
    st = dsq_inputs.Stack("wide", bits, 16, (28, 28, 64), 0.0, 2.0, None)
    st.layers = [
        Layer("a", "conv", "in", "a", 64, 64, 3, 1, 1, None, 0.0, 2.5),        # window, 64-byte rows
        Layer("e", "conv", "a", "e", 64, 256, 1, 1, 0, None, 0.0, 6.0, True),  # 1x1
        Layer("d", "dw", "e", "d", 256, 256, 3, 1, 1, None, 0.0, 6.0, True),
        Layer("p", "conv", "d", "p", 256, 128, 1, 1, 0, None, 0.0, 6.0, True),
        Layer("w", "conv", "p", "w", 128, 128, 3, 1, 1, "p", 0.0, 2.0),        # window, residual
        Layer("q", "pool", "w", "q"),
        Layer("s", "conv", "w", "s", 128, 256, 3, 2, 1, None, 0.0, 3.0),       # strided: im2col
        Layer("k", "conv", "s", "k", 256, 256, 3, 1, 1, None, 0.0, 3.0),
    ]
    st.out = "k"
    return st


# as chosen; the window kernel wherever it fits and nothing on the kernel for little work
@pytest.mark.parametrize("hook", [1, 3])
@pytest.mark.parametrize("make", [wide_stack, lambda bits: dsq_inputs.tiny_stack(bits=bits)])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_rewritten_between_passes(bits, make, hook):
    import paper_1908_05033_b200 as dsq
    from paper_1908_05033_b200.stack import GpuStack
    st = make(bits)
    dsq.dsq_set_conv3_window(hook)
    try:
        nets = [GpuStack(st, dsq_inputs.stack_params(st, workload_id=w)) for w in (9, 10)]
        x = T(dsq_inputs.stack_input(st, batch=st.batch, workload_id=9))
        want = []
        for net in nets:
            net.forward(x)
            want.append({k: v.clone() for k, v in net.codes.items()})
        assert not torch.equal(want[0][st.out], want[1][st.out])
        sources = [[{k: w[k].clone() for k in ("blob", "scale", "bias")} if w else None
                    for _, w in net.layers] for net in nets]
        net, got = nets[0], []
        for i in range(24):                      # one by one, then as a graph
            which = (i // 2 + i) % 2
            for (_, w), new in zip(net.layers, sources[which]):
                for k in new or ():
                    w[k].copy_(new[k])
            net.forward(x if i % 3 else None)    # (None: the input's codes as they are)
            got.append((which, {k: v.clone() for k, v in net.codes.items()}))
        for i, (which, codes) in enumerate(got):
            for k, v in codes.items():
                assert torch.equal(v, want[which][k]), (i, k)
        net.check()
    finally:
        dsq.dsq_set_conv3_window(1)
