"""Run a layer stack (dsq_inputs.Stack) through the C-ABI library.

Marshalling only: weights are packed once with dsq_pack_weights, every tensor
is a pre-allocated packed-code buffer, and a forward pass is one
dsq_quantize_act followed by one dsq_conv2d / dsq_dwconv2d / dsq_maxpool2x2
call per layer on the current stream.  No fp32 activation tensor is written
between layers.  The call sequence can be captured in a CUDA graph.

The layers' calls are the same in every pass, so they are made once, recorded
as finished launches, and a pass replays them from native code (2 us a launch
instead of 13 us a call; at small batch the calls took longer than the kernels).
The third pass makes a CUDA graph of them, which takes about 0.3 ms of host time once
and whatever memory CUDA keeps for a graph; later passes launch that graph.
"""
import numpy as np
import torch

from . import binding as B


def _delta_f32(bits, lo, hi):
    return (np.float32(hi) - np.float32(lo)) / np.float32(2 ** bits - 1)


class GpuStack:
    _plan = None          # the recorded pass: of this object and process only
    _packed_by = None     # version of the library that packed the weight blobs

    def __init__(self, st, params, batch=None, w_offset=0.5, device="cuda",
                 keep_debug=False):
        self.st, self.bits, self.w_offset = st, st.bits, w_offset
        self.batch = st.batch if batch is None else batch
        self.device = device
        self.keep_debug = keep_debug
        self.ws = B.new_workspace(device)
        bits = self.bits
        shapes = st.tensor_shapes()
        self.shapes = shapes
        self.ranges = {"in": (st.in_lo, st.in_hi)}
        self.codes = {}
        for name, (H, W, Cc) in shapes.items():
            self.codes[name] = torch.zeros(
                (self.batch, H, W, B.dsq_row_pitch(Cc, bits)),
                dtype=torch.uint8, device=device)
        self.layers = []
        for L in st.layers:
            if L.kind == "pool":
                self.ranges[L.dst] = self.ranges[L.src]
                self.layers.append((L, None))
                continue
            p = params[L.name]
            a_lo, a_hi = self.ranges[L.src]
            w = torch.from_numpy(p["w"]).to(device)
            per_ch = p["w_hi"].size > 1
            if per_ch:
                lo = torch.from_numpy(p["w_lo"]).to(device)
                hi = torch.from_numpy(p["w_hi"]).to(device)
            else:
                lo, hi = float(p["w_lo"][0]), float(p["w_hi"][0])
            blob, conv = B.dsq_pack_weights(w, bits, lo, hi, self.ws,
                                            depthwise=(L.kind == "dw"),
                                            stride=L.stride, pad=L.pad)
            da = _delta_f32(bits, a_lo, a_hi)
            w_lo = np.broadcast_to(p["w_lo"], (L.cout,)).astype(np.float32)
            w_hi = np.broadcast_to(p["w_hi"], (L.cout,)).astype(np.float32)
            dw = ((w_hi - w_lo) / np.float32(2 ** bits - 1)).astype(np.float32)
            scale = torch.from_numpy((da * dw).astype(np.float32)).to(device)
            bias = torch.from_numpy(p["bias"]).to(device)
            self.ranges[L.dst] = (L.out_lo, L.out_hi)
            self.layers.append((L, dict(blob=blob, conv=conv, scale=scale,
                                        bias=bias)))
        B.check_workspace(self.ws, "dsq_pack_weights")
        self._packed_by = B.dsq_version()
        self.debug = {}

    def __getstate__(self):
        """A copied or pickled stack records its own pass."""
        return {k: v for k, v in self.__dict__.items() if k != "_plan"}

    def __setstate__(self, state):
        """A stack stored by another version of the library packs its weights again."""
        self.__dict__.update(state)
        if self._packed_by != B.dsq_version() and self.ws.is_cuda:
            with torch.cuda.device(self.ws.device):
                self._pack_again()

    def _pack_again(self):
        """The packed rows at the start of a blob are a public format, the expanded copy behind
        them is its version's own: new blobs from the codes of the rows (a code q is
        what q on the range [0, 2^b - 1] quantises to)."""
        for L, w in self.layers:
            if w is None or L.kind == "dw":               # (no copy behind these rows)
                continue
            c = w["conv"]
            rows, pitch = c.Cout * c.KH * c.KW, B.dsq_row_pitch(c.Cin, self.bits)
            codes = B.dsq_unpack(w["blob"][:rows * pitch].view(rows, pitch), rows, c.Cin, self.bits, True)
            q = codes.view(c.Cout, c.KH, c.KW, c.Cin).float() + 2 ** (self.bits - 1)
            w["blob"], _ = B.dsq_pack_weights(q, self.bits, 0.0, 2 ** self.bits - 1, self.ws, stride=c.stride,
                                              pad=c.pad)
        # (usable on every stream at once, as a new stack is)
        torch.cuda.current_stream().synchronize()
        self._packed_by = B.dsq_version()

    def _parts(self):
        """Everything _call_layers reads.  Exchange one of these objects, or change a
        layer's attributes or geometry in place, and the calls are recorded again."""
        return (self.layers, self.codes, self.ranges, self.shapes, self.ws, self.batch, self.bits,
                self.w_offset)

    def forward(self, x):
        """x: fp32 NHWC CUDA tensor, or None to run the layers on the input
        codes already in place.  Returns the packed codes of st.out."""
        st = self.st
        if x is not None:
            B.dsq_quantize_act(x, self.bits, st.in_lo, st.in_hi, out=self.codes["in"])
        if self.keep_debug:                     # new output tensors in every pass
            self._call_layers()
        elif self._plan is None or not B._host.plan_run(self._plan, self._parts()):
            self._plan = B._host.plan_record(self._call_layers, self._parts())
            if not B._host.plan_run(self._plan, None):
                self._call_layers()             # (a hook was set in between)
        return self.codes[st.out]

    def _call_layers(self):
        bits = self.bits
        for L, w in self.layers:
            H, W, Cc = self.shapes[L.src]
            shape = (self.batch, H, W, Cc)
            src = self.codes[L.src]
            if L.kind == "pool":
                B.dsq_maxpool2x2(src, shape, bits, out=self.codes[L.dst])
                continue
            a_lo, a_hi = self.ranges[L.src]
            res = res_q = None
            if L.residual is not None:
                res = self.codes[L.residual]
                res_q = (bits,) + tuple(self.ranges[L.residual])
            kw = dict(w_offset=self.w_offset, residual=res, residual_q=res_q,
                      requant=(bits, L.out_lo, L.out_hi),
                      want_f32=self.keep_debug, want_acc=self.keep_debug,
                      out_codes=self.codes[L.dst])
            if L.kind == "dw":
                _, y, acc = B.dsq_dwconv2d(src, shape, (bits, a_lo, a_hi),
                                           w["blob"], w["conv"], w["scale"],
                                           w["bias"], **kw)
            else:
                _, y, acc = B.dsq_conv2d(src, shape, (bits, a_lo, a_hi),
                                         w["blob"], w["conv"], w["scale"],
                                         w["bias"], self.ws, **kw)
            if self.keep_debug:
                self.debug["y:" + L.name] = y
                self.debug["acc:" + L.name] = acc

    def n_launches(self):
        """Kernels launched by one forward pass."""
        return 1 + len(self.layers)

    def unpack(self, name):
        """int8 codes [batch, H, W, C] of a tensor (test aid)."""
        H, W, Cc = self.shapes[name]
        rows = self.batch * H * W
        return B.dsq_unpack(self.codes[name].view(rows, -1), rows, Cc,
                            self.bits, False).view(self.batch, H, W, Cc)

    def check(self):
        B.check_workspace(self.ws, "stack forward")
