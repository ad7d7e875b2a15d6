"""A stack's recorded pass: the same codes as the calls it was made from, in the passes
that launch one by one, from the graph, in a caller's capture, and after something the
calls were made from has been exchanged."""
import pytest
import torch

pytestmark = pytest.mark.gpu

import dsq_inputs
from gpu_util import T


@pytest.mark.parametrize("bits", [2, 3, 4])
def test_replayed_pass(bits):
    import paper_1908_05033_b200 as dsq
    from paper_1908_05033_b200.stack import GpuStack
    st = dsq_inputs.tiny_stack(bits=bits)
    params = dsq_inputs.stack_params(st, workload_id=9)
    calls = GpuStack(st, params, keep_debug=True)
    replay = GpuStack(st, params)
    x0 = T(dsq_inputs.stack_input(st, batch=st.batch, workload_id=9))

    def same(scale):
        want = calls.forward(x0 * scale).clone()
        assert torch.equal(replay.forward(x0 * scale), want), scale

    for i in range(6):                       # from the third run on as a graph
        same(1.0 + 0.1 * i)
    for name in ("in", st.out):              # new buffers
        replay.codes[name] = torch.zeros_like(replay.codes[name])
        for i in range(5):
            same(0.7 + 0.1 * i)
    dsq.dsq_set_dependent_launch(0)          # another way of launching
    try:
        same(0.9)
    finally:
        dsq.dsq_set_dependent_launch(1)
    x = x0.clone()
    graph = torch.cuda.CUDAGraph()
    replay.forward(x)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        out = replay.forward(x)
    x.copy_(x0 * 1.3)
    graph.replay()
    assert torch.equal(out, calls.forward(x0 * 1.3))
