"""Performance cases: the work a user of this library has it do.

A case is a dict of plain values; `kind` says which entry points it goes
through:
  stack  a quantised network through GpuStack.forward: fp32 activations in,
         packed codes of the last layer out (the deployed model, inference)
  layer  one quantised convolution on fp32 activations: dsq_quantize_act then
         dsq_conv2d (the paper's per-layer timings)
  gemm   dsq_gemm on packed codes
  bgemm  dsq_binary_gemm on packed sign bits
  wgemm  dsq_wgemm_bf16: bf16 activations times packed low-bit weights
  soft   the training side: the soft quantiser forward and backward

`listed()` are fixed cases, `draw(rng)` gives more of the same ranges,
`prepare` makes what a program holds before the call (inputs, packed weights,
workspaces), `run` is one pass, `work` the bytes and operations the pass
cannot do without, `tolerance` how far another correct implementation may be.
"""
import math

import torch

import dsq_inputs
import paper_1908_05033_b200 as dsq
from paper_1908_05033_b200.stack import GpuStack

STACKS = {"resnet18": dsq_inputs.resnet18_stack,
          "mobilenetv2": dsq_inputs.mobilenetv2_stack,
          "vgg16": dsq_inputs.vgg16_stack}


def listed():
    return [
        # one image through the ResNet-18-shaped network: interactive
        # inference, where every layer is small and latency counts
        dict(name="resnet18_b4_batch1", kind="stack", net="resnet18", bits=4, batch=1, hw=56),
        # the headline workload: the same network at the benchmark's batch
        dict(name="resnet18_b4_batch64", kind="stack", net="resnet18", bits=4, batch=64, hw=56),
        # depthwise-separable network: 1x1 convolutions around depthwise 3x3
        dict(name="mobilenetv2_b4_batch64", kind="stack", net="mobilenetv2", bits=4, batch=64,
             hw=112),
        # the largest: wide 3x3 convolutions on large images, 2-bit, with pools
        dict(name="vgg16_b2_batch32", kind="stack", net="vgg16", bits=2, batch=32, hw=224),
        # a single small convolution, fp32 in and fp32 out: the smallest call
        dict(name="conv3x3_64x56_b4_batch1", kind="layer", cin=64, cout=64, hw=56, batch=1,
             ksize=3, stride=1, bits=4, out="f32"),
        # plain GEMM sweep, smallest size: int32 result and its dequantised form
        dict(name="gemm_1024_b2", kind="gemm", m=1024, n=1024, k=1024, bits=2, out="both"),
        # plain GEMM sweep, the size the library is judged at
        dict(name="gemm_4096_b4", kind="gemm", m=4096, n=4096, k=4096, bits=4, out="i32"),
        # ragged sizes, nothing a multiple of a tile, 3-bit, dequantised result
        dict(name="gemm_2500x1111x1777_b3", kind="gemm", m=2500, n=1111, k=1777, bits=3,
             out="f32"),
        # a 3x3 convolution over 512 channels on 16 images of 14x14, binarised
        # and lowered to a GEMM (K = 9 * 512)
        dict(name="bgemm_3136x512x4608", kind="bgemm", m=3136, n=512, k=4608, out="i32"),
        # weight-only linear layer on a handful of rows (a serving step)
        dict(name="wgemm_16x4096x4096_w4", kind="wgemm", m=16, n=4096, k=4096, bits=4),
        # the same layer on many rows (a whole prompt or a training batch)
        dict(name="wgemm_2048x4096x4096_w3", kind="wgemm", m=2048, n=4096, k=4096, bits=3),
        # training: one activation tensor of the ResNet-18-shaped network
        # through the soft quantiser and back
        dict(name="soft_fwd_bwd_12.8M_b4", kind="soft", count=64 * 56 * 56 * 64, bits=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["stack"] * 4 + ["layer"] * 2 + ["gemm"] * 3 + ["bgemm"] + ["wgemm"] * 2
                      + ["soft"])
    if kind == "stack":
        net = rng.choice(sorted(STACKS))
        if net == "resnet18":
            return dict(kind=kind, net=net, bits=rng.choice([2, 3, 4]),
                        batch=_log_int(rng, 1, 64), hw=rng.randint(28, 60))
        if net == "mobilenetv2":
            return dict(kind=kind, net=net, bits=rng.choice([2, 3, 4]),
                        batch=_log_int(rng, 1, 64), hw=rng.randint(56, 116))
        # four 2x2 pools: the image side is a multiple of 16
        return dict(kind=kind, net=net, bits=rng.choice([2, 4]), batch=_log_int(rng, 1, 24),
                    hw=16 * rng.randint(4, 14))
    if kind == "layer":
        # channels and image sides of the stacks' layers, ragged images included
        cin, hw = rng.choice([(32, 112), (64, 56), (128, 28), (256, 14), (512, 7)])
        ksize = rng.choice([1, 3, 3])
        return dict(kind=kind, cin=cin, cout=rng.choice([cin, cin, 2 * cin]),
                    hw=rng.randint(max(3, hw // 2), hw + hw // 4), batch=_log_int(rng, 1, 64),
                    ksize=ksize, stride=rng.choice([1, 1, 2]), bits=rng.choice([2, 3, 4]),
                    out=rng.choice(["f32", "codes"]))
    if kind == "gemm":
        return dict(kind=kind, m=_log_int(rng, 128, 6144), n=_log_int(rng, 128, 6144),
                    k=_log_int(rng, 128, 6144), bits=rng.choice([2, 3, 4]),
                    out=rng.choice(["i32", "f32", "both"]))
    if kind == "bgemm":
        return dict(kind=kind, m=_log_int(rng, 128, 6144), n=_log_int(rng, 128, 6144),
                    k=_log_int(rng, 128, 6144), out=rng.choice(["i32", "f32"]))
    if kind == "wgemm":
        # rows of bf16 activations are read with 16-byte pitch: k is a multiple of 8
        return dict(kind=kind, m=_log_int(rng, 1, 4096), n=_log_int(rng, 512, 6144),
                    k=8 * _log_int(rng, 64, 768), bits=rng.choice([1, 2, 3, 4]))
    return dict(kind=kind, count=_log_int(rng, 1 << 14, 1 << 26), bits=rng.choice([2, 3, 4]))


def _stack_of(case):
    return STACKS[case["net"]](batch=case["batch"], bits=case["bits"], hw=case["hw"])


def _packed_random(gen, rows, k, bits):
    """Packed rows of uniformly random codes, spare bits zero as the format wants."""
    half = 1 << (bits - 1)
    codes = torch.randint(-half, half, (rows, k), dtype=torch.int8, device="cuda", generator=gen) \
        if bits > 1 else torch.randint(0, 2, (rows, k), dtype=torch.int8, device="cuda",
                                       generator=gen)
    return dsq.dsq_pack_codes(codes, bits)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def randn(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    def rand(*shape):
        return torch.rand(shape, device="cuda", generator=gen)

    kind = case["kind"]
    if kind == "stack":
        st = _stack_of(case)
        x = randn(st.batch, *st.in_shape).clamp_(0.0, st.in_cap)
        return dict(case=case, x=x, net=GpuStack(st, dsq_inputs.stack_params(st, workload_id=seed)))
    if kind == "layer":
        cin, cout, ks, hw, bits = (case[k] for k in ("cin", "cout", "ksize", "hw", "bits"))
        x = randn(case["batch"], hw, hw, cin).clamp_(min=0.0)
        ws = dsq.new_workspace()
        blob, conv = dsq.dsq_pack_weights(randn(cout, ks, ks, cin) * 0.05, bits, -0.1, 0.1, ws,
                                          stride=case["stride"], pad=ks // 2)
        dsq.check_workspace(ws, "dsq_pack_weights")
        levels = 2 ** bits - 1
        scale = torch.full((cout,), (2.0 / levels) * (0.2 / levels), device="cuda")
        return dict(case=case, x=x, ws=ws, blob=blob, conv=conv, scale=scale,
                    bias=randn(cout) * 0.1)
    if kind == "soft":
        # around the clip range [-1, 2] with both tails beyond it
        return dict(case=case, x=randn(case["count"]) * 1.2 + 0.5, g=randn(case["count"]))
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "gemm":
        return dict(case=case, A=_packed_random(gen, m, k, case["bits"]),
                    B=_packed_random(gen, n, k, case["bits"]),
                    row_scale=(rand(m) + 0.5) * 2.0 ** -10,
                    ws=dsq.new_gemm_workspace(m, n, k, case["bits"]))
    if kind == "bgemm":
        ws = torch.zeros(dsq.lib.dsq_binary_gemm_workspace_bytes(m, n, k), dtype=torch.uint8,
                         device="cuda")
        return dict(case=case, A=_packed_random(gen, m, k, 1), B=_packed_random(gen, n, k, 1),
                    row_scale=(rand(m) + 0.5) * 2.0 ** -10, ws=ws)
    ws = torch.zeros(dsq.lib.dsq_wgemm_workspace_bytes(n, k), dtype=torch.uint8, device="cuda")
    clip = rand(n) * 0.25 + 0.05
    return dict(case=case, X=randn(m, k).to(torch.bfloat16),
                W=_packed_random(gen, n, k, case["bits"]),
                col_scale=clip / (2 ** case["bits"] - 1), col_bias=randn(n) * 0.1, ws=ws)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "stack":
        return state["net"].forward(state["x"])
    if kind == "layer":
        bits = case["bits"]
        act = dsq.dsq_quantize_act(state["x"], bits, 0.0, 2.0)
        codes, y, _ = dsq.dsq_conv2d(act, tuple(state["x"].shape), (bits, 0.0, 2.0), state["blob"],
                                     state["conv"], state["scale"], state["bias"], state["ws"],
                                     w_offset=0.5,
                                     requant=(bits, 0.0, 2.0) if case["out"] == "codes" else None,
                                     want_f32=case["out"] == "f32")
        return codes if case["out"] == "codes" else y
    if kind == "soft":
        y = dsq.dsq_soft_quantize_fwd(state["x"], case["bits"], -1.0, 2.0, 0.2)
        gx, gp = dsq.dsq_soft_quantize_bwd(state["x"], state["g"], case["bits"], -1.0, 2.0, 0.2)
        return y, gx, gp
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "wgemm":
        return dsq.dsq_wgemm_bf16(state["X"], state["W"], m, n, k, case["bits"],
                                  state["col_scale"], state["col_bias"], ws=state["ws"])
    row_scale = None if case["out"] == "i32" else state["row_scale"]
    want_i32 = case["out"] != "f32"
    if kind == "gemm":
        return dsq.dsq_gemm(state["A"], state["B"], m, n, k, case["bits"], state["ws"],
                            row_scale=row_scale, want_i32=want_i32)
    return dsq.dsq_binary_gemm(state["A"], state["B"], m, n, k, ws=state["ws"],
                               row_scale=row_scale, want_i32=want_i32)


def work(case):
    """Inputs read once, outputs written once; 2 operations per multiply-
    accumulate (about 20 per element for the soft quantiser)."""
    kind = case["kind"]
    if kind == "stack":
        st = _stack_of(case)
        H, W, C = st.in_shape
        Ho, Wo, Co = st.tensor_shapes()[st.out]
        weights = sum(L.cout * L.ksize ** 2 * (1 if L.kind == "dw" else L.cin)
                      for L in st.layers if L.kind != "pool")
        elements = weights + st.batch * Ho * Wo * Co
        return {"bytes": st.batch * H * W * C * 4 + elements * st.bits / 8,
                "flops": 2 * st.batch * st.macs_per_image()}
    if kind == "layer":
        ks, cin, cout, bits = case["ksize"], case["cin"], case["cout"], case["bits"]
        ho = (case["hw"] + 2 * (ks // 2) - ks) // case["stride"] + 1
        outputs = case["batch"] * ho * ho * cout
        return {"bytes": case["batch"] * case["hw"] ** 2 * cin * 4 + ks * ks * cin * cout * bits / 8
                + outputs * (4 if case["out"] == "f32" else bits / 8),
                "flops": 2 * outputs * ks * ks * cin}
    if kind == "soft":
        return {"bytes": 20 * case["count"], "flops": 20 * case["count"]}
    m, n, k = case["m"], case["n"], case["k"]
    flops = 2 * m * n * k
    if kind == "wgemm":
        return {"bytes": m * k * 2 + n * k * case["bits"] / 8 + m * n * 4, "flops": flops}
    outputs = m * n * (8 if case["out"] == "both" else 4)
    return {"bytes": (m + n) * k * case.get("bits", 1) / 8 + outputs, "flops": flops}


def tolerance(case):
    # integer codes and accumulators, and one pinned binary32 multiply or fma
    # behind them; the bf16 GEMM and the soft quantiser sum in binary32
    if case["kind"] in ("wgemm", "soft"):
        return {"rel": 1e-5}
    return "exact"
