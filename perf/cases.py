"""The work a user has this library do, as cases that can be timed and compared.

A case is a dict of plain values.  Five kinds:

  layer     one LceBConv2d on packed words with load-time packed weights, optionally with the LceQuantize
            before it ("quantize": the input is the fp32 tensor), called directly or through a plan object
  network   the ImageNet-shaped body of seventeen 3x3 layers behind an RGB LceQuantize, bit-packed
            activations between the layers, float output at the end; call by call or as a CUDA graph
  residual  the four-stage block stack with the shortcut add and the next LceQuantize fused into the
            convolutions and a 2x2 binary max-pool between the stages
  host      one LceBConv2d whose tensors live in host memory (pinned), weights included
  tensor    the streaming operations around the convolutions on one activation tensor: LceQuantize,
            LceBMaxPool2d, LceDequantize and the fp32 add

Every output is a unique integer, bit or correctly rounded float, so all of them are compared exactly.
"""
from __future__ import annotations

import math

import torch

import paper_2011_09398_b200 as lce

DEVICE = "cuda:0"
PADDING = {"valid": lce.PAD_VALID, "one": lce.PAD_SAME_ONE, "zero": lce.PAD_SAME_ZERO}
OUT = {"f32": lce.OUT_FLOAT32, "bits": lce.OUT_BITPACKED}


def layer(batch, h, w, cin, cout, k=3, stride=1, pad="one", out="bits", relu=False, quantize=False, plan=False, **more):
    return dict(kind="layer", batch=batch, h=h, w=w, cin=cin, cout=cout, k=k, stride=stride, pad=pad, out=out,
                relu=relu, quantize=quantize, plan=plan, **more)


def listed():
    return [
        # The smallest call in use: one image's small layer, from its float activations to its float output.
        layer(1, 14, 14, 64, 64, out="f32", quantize=True, name="quantize_conv_14x14x64_b1"),
        # A ResNet-18 stage-1 layer on a serving batch; its float output is what it mostly moves.
        layer(64, 56, 56, 64, 64, out="f32", name="conv_56x56x64_b64_f32"),
        # A stage-3 layer between two binary layers, prepared once and run many times.
        layer(64, 14, 14, 256, 256, plan=True, name="conv_14x14x256_b64_bits_plan"),
        # A stage transition: stride 2.
        layer(64, 28, 28, 256, 256, stride=2, name="conv_28x28x256_s2_b64_bits"),
        # A large filter whose taps do not fit on the chip at once, and channels that do not fill their last block.
        layer(64, 32, 32, 160, 160, k=5, out="f32", name="conv_32x32x160_k5_b64_f32"),
        # A model that was not designed around 32-channel words: odd image, odd channels, zero padding, ReLU, few images.
        layer(3, 37, 29, 100, 72, pad="zero", out="f32", relu=True, name="conv_37x29x100_b3_zero_relu"),
        # One image through a network, the paper's own setting: call by call ...
        dict(kind="network", batch=1, size=224, graph=False, name="network_b1"),
        # ... and captured once and replayed, as a latency-bound server runs it.
        dict(kind="network", batch=1, size=224, graph=True, name="network_b1_graph"),
        # The same network at throughput batch.
        dict(kind="network", batch=256, size=224, graph=False, name="network_b256"),
        # Shortcut blocks (float residual path beside the binary one).
        dict(kind="residual", batch=128, size=56, name="residual_b128"),
        # A caller whose tensors live in host memory.
        dict(kind="host", batch=64, h=28, w=28, cin=128, cout=128, k=3, stride=1, pad="one", out="bits", name="host_conv_28x28x128_b64_bits"),
        # The streaming operations on one activation tensor larger than the L2.
        dict(kind="tensor", batch=128, h=56, w=56, c=128, name="tensor_ops_56x56x128_b128"),
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _channels(rng):
    # mostly whole words, as models are built; sometimes not
    c = _log(rng, 32, 512)
    return c if rng.random() < 0.25 else max(32, (c + 16) // 32 * 32)


def _conv_shape(rng, most_macs):
    while True:
        c = dict(batch=_log(rng, 1, 64), h=_log(rng, 7, 64), w=0, cin=_channels(rng), cout=0, k=rng.choice([3, 3, 3, 3, 1, 5]),
                 stride=rng.choice([1, 1, 1, 2]), pad=rng.choice(["one", "one", "one", "zero", "valid"]), out=rng.choice(["f32", "bits"]))
        c["w"] = c["h"] if rng.random() < 0.7 else _log(rng, 7, 64)
        c["cout"] = c["cin"] if rng.random() < 0.5 else _channels(rng)
        oh, ow = _extent(c["h"], c), _extent(c["w"], c)
        if c["batch"] * oh * ow * c["cout"] * c["k"] ** 2 * c["cin"] <= most_macs:
            return c


def draw(rng):
    kind = rng.choice(["layer"] * 6 + ["network", "network", "residual", "host", "tensor"])
    if kind == "layer":
        c = _conv_shape(rng, 2 ** 38)
        return layer(**c, relu=c["out"] == "f32" and rng.random() < 0.3, quantize=rng.random() < 0.2, plan=rng.random() < 0.3)
    if kind == "network":
        size = _log(rng, 96, 256)
        return dict(kind=kind, batch=_log(rng, 1, 256 * 224 * 224 // max(size, 224) ** 2), size=size, graph=rng.random() < 0.5)
    if kind == "residual":
        return dict(kind=kind, batch=_log(rng, 1, 128), size=_log(rng, 24, 56))
    if kind == "host":
        return dict(kind=kind, **_conv_shape(rng, 2 ** 34))
    c = _log(rng, 3, 512)
    h, w = _log(rng, 7, 112), _log(rng, 7, 112)
    return dict(kind=kind, batch=_log(rng, 1, max(1, min(256, 128 * 56 * 56 * 128 // (h * w * c)))), h=h, w=w, c=c)


# --- inputs ------------------------------------------------------------------------------------


def _extent(size, c):
    return (size - c["k"]) // c["stride"] + 1 if c["pad"] == "valid" else -(-size // c["stride"])


def _words(c):
    return (c + 31) // 32


class Draws:
    """Activations ~N(0,1), weights uniform +-1, multipliers ~U(0.5,1.5), biases ~N(0,0.1), thresholds ~rint(N(0,sqrt K))."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEVICE).manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEVICE)

    def weights(self, *shape):
        return lce.pack_weights(torch.randint(0, 2, shape, generator=self.g, device=DEVICE, dtype=torch.int8) * 2 - 1)

    def transform(self, cout, K, out):
        """(multiplier, bias, thresholds) of a layer, None where its output type has no use for them."""
        if out == "bits":
            return None, None, torch.round(self.normal(cout) * math.sqrt(K)).to(torch.int32)
        return torch.rand(cout, generator=self.g, device=DEVICE) + 0.5, self.normal(cout) * 0.1, None


def _conv(draws, batch, h, w, cin, cout, k=3, stride=1, pad="one", out="bits", relu=False):
    """(descriptor, packed weights, multiplier, bias, thresholds) of a layer as a loaded model keeps them."""
    desc = lce.make_desc(batch, h, w, cin, cout, (k, k), (stride, stride), PADDING[pad], OUT[out],
                         lce.ACT_RELU if relu else lce.ACT_NONE, weights_packed=1)
    return (desc, lce.lce_bconv2d_pack_weights(desc, draws.weights(cout, k, k, cin)), *draws.transform(cout, k * k * cin, out))


def _network_shapes(case):
    """(side, cin, cout, stride, out) of the seventeen layers."""
    h, c, shapes = case["size"], 3, []
    for width, count in ((32, 1), (64, 4), (128, 4), (256, 4), (512, 4)):
        for i in range(count):
            stride = 2 if i == 0 else 1
            shapes.append((h, c, width, stride, "bits"))
            h, c = -(-h // stride), width
    shapes[-1] = shapes[-1][:4] + ("f32",)
    return shapes


RESIDUAL_WIDTHS = (64, 128, 256, 512)


def _output(case, h, w, cout, out):
    n = case["batch"]
    return torch.empty((n, h, w, _words(cout)), dtype=torch.int32, device=DEVICE) if out == "bits" else torch.empty((n, h, w, cout), device=DEVICE)


def prepare(case, seed):
    d = Draws(seed)
    n, kind = case["batch"], case["kind"]
    if kind == "layer":
        conv = _conv(d, *(case[x] for x in ("batch", "h", "w", "cin", "cout", "k", "stride", "pad", "out", "relu")))
        x = d.normal(n, case["h"], case["w"], case["cin"])
        if not case["quantize"]:
            x = lce.lce_bitpack(x)
        state = dict(kind="plan" if case["plan"] else "layer", quantize=case["quantize"], x=x, conv=conv)
        if case["plan"]:
            state["packed"] = torch.empty((n, case["h"], case["w"], _words(case["cin"])), dtype=torch.int32, device=DEVICE) if case["quantize"] else x
            state["plan"] = lce.lce_bconv2d_plan_create(conv[0], state["packed"], *conv[1:])
        return state
    if kind == "network":
        x = d.normal(n, case["size"], case["size"], 3)
        state = dict(kind="calls", x=x, first=torch.empty((n, case["size"], case["size"], 1), dtype=torch.int32, device=DEVICE), layers=[])
        for h, cin, cout, stride, out in _network_shapes(case):
            state["layers"].append((*_conv(d, n, h, h, cin, cout, 3, stride, "one", out), _output(case, -(-h // stride), -(-h // stride), cout, out)))
        if case["graph"]:
            _network(state)
            torch.cuda.synchronize()
            state["graph"] = torch.cuda.CUDAGraph()
            with torch.cuda.graph(state["graph"]):
                _network(state)
            state["kind"] = "graph"
        return state
    if kind == "residual":
        h, stages = case["size"], []
        state = dict(kind="residual", x=d.normal(n, h, h, RESIDUAL_WIDTHS[0]), stages=stages)
        state["a"] = _output(case, h, h, RESIDUAL_WIDTHS[0], "bits")
        for i, c in enumerate(RESIDUAL_WIDTHS):
            s = dict(conv1=_conv(d, n, h, h, c, c), conv2=_conv(d, n, h, h, c, c, out="f32"), b=_output(case, h, h, c, "bits"), y=None, p=None, trans=None)
            if i + 1 < len(RESIDUAL_WIDTHS):
                s["p"], wide = _output(case, h, h, c, "bits"), RESIDUAL_WIDTHS[i + 1]
                h //= 2
                s.update(q=_output(case, h, h, c, "bits"), trans=_conv(d, n, h, h, c, wide, k=1, out="f32"), x=_output(case, h, h, wide, "f32"), a=_output(case, h, h, wide, "bits"))
            else:
                s["y"] = _output(case, h, h, c, "f32")
            stages.append(s)
        return state
    if kind == "host":
        desc = lce.make_desc(n, case["h"], case["w"], case["cin"], case["cout"], (case["k"],) * 2, (case["stride"],) * 2, PADDING[case["pad"]], OUT[case["out"]])
        x = lce.lce_bitpack(d.normal(n, case["h"], case["w"], case["cin"]))
        w = d.weights(case["cout"], case["k"], case["k"], case["cin"])
        tensors = [t if t is None else t.cpu().pin_memory() for t in (x, w, *d.transform(case["cout"], case["k"] ** 2 * case["cin"], case["out"]))]
        out = _output(case, _extent(case["h"], case), _extent(case["w"], case), case["cout"], case["out"]).cpu().pin_memory()
        return dict(kind="host", args=(desc, *tensors, out, torch.empty(lce.lce_bconv2d_host_workspace_bytes(desc), dtype=torch.uint8, device=DEVICE)), out=out)
    shape = (n, case["h"], case["w"], case["c"])
    return dict(kind="tensor", channels=case["c"], a=d.normal(*shape), b=d.normal(*shape))


# --- one pass ----------------------------------------------------------------------------------


def _network(state):
    x = lce.lce_bitpack(state["x"], state["first"])
    for desc, w, mult, bias, thr, out in state["layers"]:
        x = lce.lce_bconv2d(desc, x, w, mult, bias, thr, out)
    return x


def _residual(state):
    x, a = state["x"], lce.lce_bitpack(state["x"], state["a"])
    for s in state["stages"]:
        desc, w, mult, bias, thr = s["conv1"]
        b = lce.lce_bconv2d(desc, a, w, mult, bias, thr, s["b"])
        desc, w, mult, bias, _ = s["conv2"]
        lce.lce_bconv2d_fused(desc, b, w, mult, bias, x, s["y"], s["p"])
        if s["trans"] is None:
            return s["y"]
        desc, w, mult, bias, _ = s["trans"]
        q = lce.lce_bmaxpool(s["p"], desc.in_c, (2, 2), (2, 2), lce.PAD_VALID, s["q"])
        x, a = s["x"], s["a"]
        lce.lce_bconv2d_fused(desc, q, w, mult, bias, None, x, a)


def run(state):
    kind = state["kind"]
    if kind == "layer":
        x = lce.lce_bitpack(state["x"]) if state["quantize"] else state["x"]
        desc, w, mult, bias, thr = state["conv"]
        return lce.lce_bconv2d(desc, x, w, mult, bias, thr)
    if kind == "plan":
        if state["quantize"]:
            lce.lce_bitpack(state["x"], state["packed"])
        return lce.lce_plan_run(state["plan"])
    if kind == "calls":
        return _network(state)
    if kind == "graph":
        state["graph"].replay()
        return state["layers"][-1][-1]
    if kind == "residual":
        return _residual(state)
    if kind == "host":
        lce.lce_bconv2d_host(*state["args"])
        return state["out"]
    words = lce.lce_bitpack(state["a"])
    return (words, lce.lce_bmaxpool(words, state["channels"]), lce.lce_unpack(words, state["channels"]), lce.lce_add_f32(state["a"], state["b"]))


# --- what a pass cannot do without -------------------------------------------------------------


def _conv_macs(n, oh, ow, cin, cout, k):
    return n * oh * ow * cout * k * k * cin


def _conv_bytes(cin, cout, k, out):
    """Weights at one bit each and the per-channel arrays."""
    return 4 * cout * k * k * _words(cin) + (4 if out == "bits" else 8) * cout


def _out_bytes(n, oh, ow, cout, out):
    return 4 * n * oh * ow * (_words(cout) if out == "bits" else cout)


def work(case):
    """Bytes: inputs and constants once, outputs once (nothing for what stays inside a chain of layers).  Operations: two per binary MAC."""
    n, kind = case["batch"], case["kind"]
    if kind in ("layer", "host"):
        h, w, cin, cout, k, out = (case[x] for x in ("h", "w", "cin", "cout", "k", "out"))
        oh, ow = _extent(h, case), _extent(w, case)
        read = 4 * n * h * w * (cin if case.get("quantize") else _words(cin)) + _conv_bytes(cin, cout, k, out)
        return {"bytes": read + _out_bytes(n, oh, ow, cout, out), "flops": 2 * _conv_macs(n, oh, ow, cin, cout, k)}
    if kind == "network":
        total, macs = 4 * n * case["size"] ** 2 * 3, 0
        for h, cin, cout, stride, out in _network_shapes(case):
            oh = -(-h // stride)
            total += _conv_bytes(cin, cout, 3, out)
            macs += _conv_macs(n, oh, oh, cin, cout, 3)
        return {"bytes": total + _out_bytes(n, oh, oh, cout, out), "flops": 2 * macs}
    if kind == "residual":
        h, total, macs = case["size"], 4 * n * case["size"] ** 2 * RESIDUAL_WIDTHS[0], 0
        for i, c in enumerate(RESIDUAL_WIDTHS):
            total += _conv_bytes(c, c, 3, "bits") + _conv_bytes(c, c, 3, "f32")
            macs += 2 * _conv_macs(n, h, h, c, c, 3)
            if i + 1 < len(RESIDUAL_WIDTHS):
                h //= 2
                total += _conv_bytes(c, RESIDUAL_WIDTHS[i + 1], 1, "f32")
                macs += _conv_macs(n, h, h, c, RESIDUAL_WIDTHS[i + 1], 1)
        return {"bytes": total + _out_bytes(n, h, h, c, "f32"), "flops": 2 * macs}
    pixels, c = n * case["h"] * case["w"], case["c"]
    pooled = n * max(0, (case["h"] - 2) // 2 + 1) * max(0, (case["w"] - 2) // 2 + 1)
    return {"bytes": 4 * (2 * pixels * c + 2 * pixels * c + (pixels + pooled) * _words(c)), "flops": 2 * pixels * c}


def tolerance(case):
    return "exact"
