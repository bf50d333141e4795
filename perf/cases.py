"""What the performance of this framework is measured on: the calls a quantization-aware training or an
inference program makes, from the smallest activation tensor to the largest, through the public entry points.

Every case is one `kind` of work with its sizes:

  fused    range, quantize, dequantize and straight-through gradient of one tensor in one call
  forward  the same without a gradient (inference, calibration of the next layer)
  train    a layer in a training step: the forward pass keeps the mask at one bit per element, the backward pass
           runs from the mask; outputs are new tensors on every step, as a training loop needs them
  shared   a layer of the batch-sharded step: range, (exchange,) forward with that range, backward from the mask
  set      the activation tensors of a whole small network in one host call
  weights  all weight tensors of a network, per output channel, in one launch
  integer  a pointwise layer on integer codes: encode the activation, accumulate over the codes
  store    an activation kept as packed codes and expanded again: encode, decode
  stats    fake quantization with the distortion sums of Table 2, layer-wise or channel-wise

Activations are [N, C, H, W] (or [N, H, W, C] with layout "nhwc"); values follow `workloads.py`: post-ReLU
half-normal with a log-normal spread per channel, or signed heavy-tailed ones, the gradient standard normal.
"""
import math

import torch

from paper_2503_18339_b200 import binding as g
from paper_2503_18339_b200 import data_parallel
from paper_2503_18339_b200.workloads import config_tensors, weight_shapes

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
GROUPS = {"channel": g.GROUP_CHANNEL, "sample": g.GROUP_SAMPLE_CHANNEL, "tensor": g.GROUP_TENSOR}


def _act(name, kind, n, c, h, w, bits, dtype="f32", values="relu", group="channel", layout="nchw", **more):
    """n, c, h, w are the dims as stored: with layout "nhwc" the channel is the last of them."""
    return dict(name=name, kind=kind, n=n, c=c, h=h, w=w, bits=bits, dtype=dtype, values=values, group=group,
                layout=layout, **more)


def listed():
    return [
        # the first layer of a small network at batch 16: one call of latency, 1 MB
        _act("first_layer", "fused", 16, 16, 32, 32, 3),
        # the 19 activation tensors of the small network at batch 256, forward and backward in one host call
        dict(name="small_network_set", kind="set", n=256, bits=4, dtype="f32", values="relu"),
        # a layer of a training step, early in an ImageNet-sized network
        _act("train_layer_56", "train", 128, 64, 56, 56, 4),
        # the largest activation of the benchmark, forward and backward
        _act("fused_112", "fused", 128, 96, 112, 112, 4, values="relu"),
        # inference in bf16 at 8 bits, signed heavy-tailed activations
        _act("forward_bf16_28", "forward", 256, 512, 28, 28, 8, dtype="bf16", values="heavy"),
        # thin planes late in a mobile network, range exchanged between data-parallel ranks
        _act("shared_range_7", "shared", 128, 960, 7, 7, 5),
        # an activation stored channels-last, bf16, forward and backward
        _act("channels_last_bf16", "fused", 128, 28, 28, 192, 4, dtype="bf16", layout="nhwc"),
        # odd planes and an odd number of channels: slabs that are not whole 16-byte units
        _act("ragged_27", "fused", 100, 75, 27, 27, 5),
        # a pointwise layer on 4-bit codes: encode, then accumulate to as many output channels
        _act("integer_layer_14", "integer", 128, 256, 14, 14, 4, out=256),
        # activations kept in memory as 5-bit codes: encode on the way forward, decode when needed again
        _act("code_store_56", "store", 128, 144, 56, 56, 5),
        # all weight tensors of an ImageNet-sized network, per output channel
        dict(name="network_weights", kind="weights", net="resnet18", first=0, count=21, bits=4, dtype="f32", grad=False),
        # the layer-wise baseline of Table 2 with its distortion sums
        _act("layerwise_stats", "stats", 128, 128, 28, 28, 4, group="tensor"),
    ]


MAX_ELEMENTS = 128 * 96 * 112 * 112


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _plane(rng, most=112):
    """Height and width: the usual sizes, or any (odd ones among them)."""
    usual = [s for s in (7, 8, 14, 16, 28, 32, 56, 112) if s <= most]
    if rng.random() < 0.6:
        s = rng.choice(usual)
        return s, s
    s = _log_uniform(rng, 5, most)
    return s, max(5, min(most, s + rng.choice((-1, 0, 0, 1))))


def draw(rng):
    kind = rng.choice(("fused", "fused", "fused", "forward", "forward", "train", "train", "shared", "set", "weights", "integer",
                       "store", "stats"))
    bits = rng.randint(2, 8)
    return _unnamed(_draw_kind(rng, kind, bits))


def _draw_kind(rng, kind, bits):
    if kind == "set":
        return dict(kind="set", n=_log_uniform(rng, 32, 320), bits=bits, dtype=rng.choice(("f32", "f32", "bf16")),
                    values="relu")
    if kind == "weights":
        net = rng.choice(("resnet20", "resnet18"))
        grad = rng.random() < 0.5
        have = len(weight_shapes(net))
        count = rng.randint(6, 16 if grad else min(have, 21))
        return dict(kind="weights", net=net, first=rng.randint(0, have - count), count=count, bits=bits,
                    dtype=rng.choice(("f32", "f32", "bf16")), grad=grad)
    dtype = rng.choice(("f32", "f32", "bf16"))
    layout, group = "nchw", "channel"
    h, w = _plane(rng, 56 if kind in ("integer", "stats", "store") else 112)
    if kind in ("fused", "forward"):
        if rng.random() < 0.2:
            layout = "nhwc"
        elif rng.random() < 0.25:
            group = rng.choice(("sample", "tensor"))
    elif kind == "stats":
        group = rng.choice(("channel", "sample", "tensor"))
    # elements spread over their logarithm, then batch and channels to match
    # (an integer layer up to the size of the listed pointwise layers of the benchmark)
    most = {"fused": MAX_ELEMENTS, "forward": MAX_ELEMENTS, "integer": 26_000_000}.get(kind, MAX_ELEMENTS // 2)
    want = _log_uniform(rng, 300_000, most)
    n = min(256, max(8, _log_uniform(rng, 8, 256)))
    if kind == "integer":
        c = max(16, min(512, want // (n * h * w))) // 16 * 16
        n = max(1, min(n, most // (c * h * w)))
        return _act(None, kind, n, c, h, w, rng.choice((4, 4, 8, bits)), dtype, group=group, layout=layout,
                    out=rng.choice((64, 128, 256)))
    c = max(3, min(2048, want // (n * h * w)))
    if rng.random() < 0.7 or layout == "nhwc":
        c = max(8, c // 8 * 8)
    n = max(1, min(n, most // (c * h * w)))
    case = _act(None, kind, n, c, h, w, bits, dtype, rng.choice(("relu", "heavy")), group, layout)
    if layout == "nhwc":
        case["c"], case["h"], case["w"] = h, w, c          # dims as stored; the channel is the last one
    return case


def _unnamed(case):
    return {k: v for k, v in case.items() if k != "name"}


def _activation(gen, shape, axis, values, dtype):
    """Values of an activation tensor: spread per channel, post-ReLU or signed heavy-tailed; finite, no -0."""
    x = torch.randn(shape, generator=gen, device="cuda")
    if values == "heavy":
        q = torch.rand(shape, generator=gen, device="cuda")
        x.mul_(q.clamp_min_(1e-3).rsqrt_())
    view = [1] * len(shape)
    view[axis] = shape[axis]
    x.mul_(torch.randn(shape[axis], generator=gen, device="cuda").mul_(0.8).exp_().view(view))
    if values == "relu":
        x.clamp_min_(0.0)
    return x.add_(0.0).to(dtype)


def prepare(case, seed):
    case = _unnamed(case)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    kind, dtype, bits = case["kind"], DTYPES[case["dtype"]], case["bits"]
    if kind == "set":
        items, outs, total = [], [], 0
        specs = [s.with_batch(case["n"]) for s in config_tensors(2)]
        for s in specs:
            x = _activation(gen, s.shape, 1, "relu", dtype)
            items.append((x, bits, torch.randn(s.shape, generator=gen, device="cuda").to(dtype)))
            total += s.shape[1]
        lo, hi = (torch.empty(total, device="cuda") for _ in range(2))       # one range buffer for the network
        at = 0
        for s in specs:
            outs.append(g.FakeQuantOut(lo=lo[at:at + s.shape[1]], hi=hi[at:at + s.shape[1]]))
            at += s.shape[1]
        return dict(kind=kind, batch=g.FusedBatch(items, outs=outs, zeroed=True), lo=lo, hi=hi)
    if kind == "weights":
        shapes = weight_shapes(case["net"])[case["first"]:case["first"] + case["count"]]
        ws, gs = [], []
        for s in shapes:
            fan_in = math.prod(s[1:])
            w = torch.randn(s, generator=gen, device="cuda").mul_(math.sqrt(2.0 / fan_in))
            w.mul_(torch.randn(s[0], generator=gen, device="cuda").mul_(0.5).exp_().view([-1] + [1] * (len(s) - 1)))
            ws.append(w.add_(0.0).to(dtype))
            gs.append(torch.randn(s, generator=gen, device="cuda").mul_(0.1).to(dtype))
        return dict(kind=kind, batch=g.WeightBatch(ws, bits, gs if case["grad"] else None))
    shape = (case["n"], case["c"], case["h"], case["w"])
    axis = 3 if case["layout"] == "nhwc" else 1
    st = dict(kind=kind, bits=bits, axis=axis, group=GROUPS[case["group"]], shape=shape, dtype=dtype)
    st["x"] = _activation(gen, shape, axis, case["values"], dtype)
    if kind in ("fused", "train", "shared"):
        st["gy"] = torch.randn(shape, generator=gen, device="cuda").to(dtype)
    if kind in ("fused", "forward", "stats"):
        # a program that meets the same layer again keeps its output buffers and its workspace
        st["out"] = g.FakeQuantOut(y=torch.empty_like(st["x"]),
                                   workspace=g.make_workspace(st["x"], axis, st["group"]))
        if kind == "fused":
            st["out"].gx = torch.empty_like(st["x"])
    if kind == "integer":
        st["weights"] = torch.randn((case["out"], case["c"]), generator=gen, device="cuda").mul_(1.0 / math.sqrt(case["c"]))
        st["out"] = g.FakeQuantOut(workspace=g.make_workspace(st["x"]))
        st["y"] = torch.empty((case["n"], case["out"], case["h"], case["w"]), device="cuda")
        st["acc_ws"] = torch.empty(g.accumulate_workspace_bytes(shape, 1, case["out"]), dtype=torch.uint8, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind == "set":
        outs = st["batch"].run()
        return [[o.y for o in outs], [o.gx for o in outs], st["lo"], st["hi"]]
    if kind == "weights":
        outs = st["batch"].run()
        return [[o.y for o in outs], [o.gx for o in outs], [o.lo for o in outs], [o.hi for o in outs]]
    x, bits, axis, group = st["x"], st["bits"], st["axis"], st["group"]
    if kind == "fused":
        o = g.granq_fakequant_fused(x, bits, gy=st["gy"], channel_axis=axis, group=group, out=st["out"])
        return [o.y, o.gx, o.lo, o.hi]
    if kind == "forward":
        o = g.granq_fakequant_fused(x, bits, channel_axis=axis, group=group, out=st["out"])
        return [o.y, o.lo, o.hi]
    if kind == "train":
        o = g.granq_fakequant_fused_fwd_packmask(x, bits, channel_axis=axis, group=group)
        gx = g.granq_fakequant_bwd_packmask(st["gy"], o.packed_mask)
        return [o.y, o.packed_mask, o.lo, o.hi, gx]
    if kind == "shared":
        o = data_parallel.fakequant_forward(x, bits, channel_axis=axis, group_mode=group)
        gx = data_parallel.fakequant_backward(st["gy"], o.packed_mask)
        return [o.y, o.packed_mask, o.lo, o.hi, gx]
    if kind == "integer":
        o = g.granq_quantize_packed_fused(x, bits, channel_axis=axis, group=group, out=st["out"])
        y, _ = g.granq_accumulate_codes(o.packed_codes, st["shape"], bits, o.s, o.z, st["weights"], y=st["y"],
                                        workspace=st["acc_ws"])
        return [y, o.packed_codes, o.s, o.z, o.lo, o.hi]
    if kind == "store":
        o = g.granq_quantize_packed_fused(x, bits, channel_axis=axis, group=group)
        y = g.granq_dequantize_packed(o.packed_codes, st["shape"], st["dtype"], bits, o.s, o.z, channel_axis=axis, group=group)
        return [y, o.packed_codes, o.s, o.z, o.lo, o.hi]
    o = g.granq_fakequant_fused_stats(x, bits, channel_axis=axis, group=group, out=st["out"])
    return [o.y, o.sums, o.lo, o.hi]


def _elements_and_groups(case):
    kind = case["kind"]
    if kind == "set":
        specs = [s.with_batch(case["n"]) for s in config_tensors(2)]
        return sum(s.numel for s in specs), sum(s.shape[1] for s in specs)
    if kind == "weights":
        shapes = weight_shapes(case["net"])[case["first"]:case["first"] + case["count"]]
        return sum(math.prod(s) for s in shapes), sum(s[0] for s in shapes)
    n, c, h, w = case["n"], case["c"], case["h"], case["w"]
    channels, outer = (w, n * c * h) if case["layout"] == "nhwc" else (c, n)
    return n * c * h * w, {"channel": channels, "sample": channels * outer, "tensor": 1}[case["group"]]


def work(case):
    """Bytes: every input read once and every output written once.  Operations: the quantizer's dozen per element
    (range, divide, add, round, clamp, scale, compare) and the multiply-adds of the pointwise layer."""
    e, groups = _elements_and_groups(case)
    kind, size, b = case["kind"], 4 if case["dtype"] == "f32" else 2, case["bits"]
    flops = 12.0 * e
    if kind in ("fused", "set") or (kind == "weights" and case["grad"]):
        nbytes = 4 * size * e                                      # x, gy -> y, gx
    elif kind in ("train", "shared"):
        nbytes = 4 * size * e + e / 8                              # x, gy -> y, gx and the mask
    elif kind == "integer":
        pixels = case["n"] * case["h"] * case["w"]
        nbytes = size * e + e * b / 8 + 4 * pixels * case["out"] + 4 * case["out"] * case["c"]
        flops += 2.0 * pixels * case["c"] * case["out"]
    elif kind == "store":
        nbytes = 2 * size * e + e * b / 8                          # x -> codes, y
    else:
        nbytes = 2 * size * e                                      # x -> y
    return {"bytes": nbytes + 8 * groups, "flops": flops}


def tolerance(case):
    """Fake quantization is defined down to the last bit: outputs are exact.  The pointwise layer multiplies scaled
    weights split into two bf16 halves (2^-17 of a weight is left out) and sums in fp32: 2.6e-6 off the same sum in
    fp64, 3.4e-5 at the worst element.  The distortion sums are fp32 partial sums of a pack, added up in fp64 in the
    order in which the blocks finish: up to 2e-8 off the sums in fp64.  Both stated about four times over."""
    if case["kind"] == "integer":
        return {"rel": 1e-5, "max": 1.4e-4}
    if case["kind"] == "stats":
        return {"rel": 8e-8, "max": 8e-8}
    return "exact"
