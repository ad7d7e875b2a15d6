"""A stack's recorded pass: the same codes as the calls it was made from, in the passes
that launch one by one, from the graph, in a caller's capture, and after something the
calls were made from has been exchanged."""
import copy
import pickle
import threading

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


def _pair(bits=4):
    """A stack that makes its calls in every pass and one that replays them, of the same
    layer list."""
    from paper_1908_05033_b200.stack import GpuStack
    st = dsq_inputs.tiny_stack(bits=bits)
    params = dsq_inputs.stack_params(st, workload_id=9)
    x = T(dsq_inputs.stack_input(st, batch=st.batch, workload_id=9))
    return GpuStack(st, params, keep_debug=True), GpuStack(st, params), x


@pytest.mark.parametrize("passes", [1, 5])       # launched one by one, and as a graph
def test_changes_in_place(passes):
    """What a layer is made of may be changed in place between two passes."""
    calls, replay, x = _pair()

    def same():
        want = calls.forward(x).clone()
        assert torch.equal(replay.forward(x), want)
        return want

    for _ in range(passes):
        before = same()
    layer = next(L for L, _ in replay.layers if L.name == "c3")      # (both stacks' layer)
    layer.out_hi = 0.7
    assert not torch.equal(before, same())
    layer.residual = None                        # no shortcut any more
    same()
    # geometry of a 1x1 convolution, a ctypes structure: a stride it does not take is refused
    for net in (calls, replay):
        next(w for L, w in net.layers if L.name == "pj")["conv"].stride = 3
    for net in (calls, replay):
        with pytest.raises(RuntimeError, match="not supported"):
            net.forward(x)
        next(w for L, w in net.layers if L.name == "pj")["conv"].stride = 1
    same()


def test_values_read_on_the_host():
    """A range held as a tensor is read in every pass, and so is a layer of a class whose
    attributes are not in its dict."""
    calls, replay, x = _pair()
    hi = torch.tensor(2.0)

    class Slots:
        __slots__ = ("name", "kind", "src", "dst", "residual", "out_lo", "out_hi")

        def __init__(self, L):
            for k in self.__slots__:
                setattr(self, k, getattr(L, k))

    for net in (calls, replay):
        i = next(i for i, (L, _) in enumerate(net.layers) if L.name == "c3")
        net.layers[i] = (Slots(net.layers[i][0]), net.layers[i][1])
        net.layers[i][0].out_hi = hi
    slots = [next(L for L, _ in net.layers if L.name == "c3") for net in (calls, replay)]
    for value in (2.0, 0.7, 1.1, 1.1):
        hi.fill_(value)
        assert torch.equal(replay.forward(x), calls.forward(x)), value
    for value in (0.8, 1.9):
        for s in slots:
            s.out_hi = value
        assert torch.equal(replay.forward(x), calls.forward(x)), value


@pytest.mark.parametrize("how", [copy.copy, copy.deepcopy, lambda net: pickle.loads(pickle.dumps(net))])
def test_copies(how):
    """A stack that has recorded its pass can still be copied and pickled; the copy gives
    the same codes from buffers of its own (a shallow one from the same)."""
    calls, replay, x = _pair()
    for passes in (1, 4):
        for _ in range(passes):
            replay.forward(x)
        other = how(replay)
        for scale in (1.0, 1.3, 0.8, 1.1):
            want = calls.forward(x * scale).clone()
            assert torch.equal(other.forward(x * scale), want)
        assert torch.equal(replay.forward(x * 0.9), calls.forward(x * 0.9))


def test_graph_made_during_a_capture_in_another_thread():
    """The third pass makes its graph while another thread captures in the mode that
    forbids most calls to every thread: the capture stands, and so do the passes."""
    calls, replay, x = _pair()
    want = calls.forward(x).clone()
    replay.forward(x)
    got = []
    stream = torch.cuda.Stream()

    def passes():
        with torch.cuda.stream(stream):
            got.extend(replay.forward(x) for _ in range(4))

    y = torch.zeros(1000, device="cuda")
    thread = threading.Thread(target=passes)
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        y += 1
        thread.start()
        thread.join()
        y += 1
    graph.replay()
    torch.cuda.synchronize()
    assert float(y[0]) == 2 and len(got) == 4
    assert torch.equal(got[-1], want)


@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("make", [lambda bits: dsq_inputs.resnet18_stack(batch=2, bits=bits, hw=14),
                                  lambda bits: dsq_inputs.tiny_stack(bits=bits)], ids=["resnet18", "every_kind"])
def test_stack_stored_by_another_version(make, bits):
    """Its blobs have the same packed rows, and behind them what this version cannot read."""
    import paper_1908_05033_b200 as dsq
    from paper_1908_05033_b200.stack import GpuStack
    st = make(bits)
    net = GpuStack(st, dsq_inputs.stack_params(st, workload_id=5))
    x = torch.randn(st.batch, *st.in_shape, device="cuda").clamp_(0.0, st.in_cap)
    weights = [w for _, w in net.layers if w is not None]
    taps = [w["conv"].KH * w["conv"].KW * (1 if w["conv"].groups > 1 else w["conv"].Cout) for w in weights]
    rows = [t * dsq.dsq_row_pitch(w["conv"].Cin, bits) for t, w in zip(taps, weights)]
    dsq.dsq_set_conv3_window(3)                  # (the kernel that reads the copy)
    try:
        want = net.forward(x).clone()
        state = pickle.loads(pickle.dumps(net)).__getstate__()
        state.pop("_packed_by")
        state["codes"][st.out].zero_()
        for n, (_, w) in zip(rows, [e for e in state["layers"] if e[1] is not None]):
            w["blob"][n:] = 0x41
        old = GpuStack.__new__(GpuStack)
        old.__setstate__(pickle.loads(pickle.dumps(state)))
        assert torch.equal(old.forward(x), want)
        old.check()
        again = [w for _, w in old.layers if w is not None]
        assert all(torch.equal(a["blob"][:n], b["blob"][:n]) for n, a, b in zip(rows, again, weights))
        # of this version: the blobs as they are
        other = pickle.loads(pickle.dumps(old))
        assert all(a is None or torch.equal(a["blob"], b["blob"])
                   for (_, a), (_, b) in zip(other.layers, old.layers))
    finally:
        dsq.dsq_set_conv3_window(1)
