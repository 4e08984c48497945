"""Timed cases of the library: the calls a user's program makes, over the sizes it makes them at.

Each case names one public entry point of ``paper_2505_03254_b200.binding`` and the sizes and options
of the call.  The channel counts are those of MobileNetV2 at its width multipliers (0.75 to 2.0) and
of the single-layer workloads of the benchmark and the tests; rows are batch * height * width of the
spatial sizes those networks pass through.  ``listed()`` are the fixed cases, ``draw()`` gives others
of the same ranges.

Inputs are what the path meets in use: activations of the post-ReLU6 distribution (uniform on
[0, 127] with 30 % zeros) or symmetric ones for layers behind a linear layer, ternary weights with
half of them zero, requantisation constants calibrated to the layer's fan-in (so that a chain of
layers keeps using the int8 range), float activations and He-normal float weights for the quantisers.
"""
import math

import torch

from paper_2505_03254_b200 import binding, synth

WIDTHS = (0.75, 1.0, 1.25, 1.4, 2.0)
#: channel counts of single layers: the networks' at widths 0.75 to 2.0 and the shape sweep's
NARROW = (16, 24, 32, 40, 48, 56, 64, 72, 96, 112, 120, 128, 144, 160, 192, 240, 320)
WIDE = (96, 144, 192, 240, 288, 336, 384, 432, 480, 576, 672, 720, 960, 1280)
SPATIAL = (7, 10, 12, 14, 20, 28, 40, 48, 56, 80, 96, 112)

#: nothing costs more than the largest listed case (1 605 632 x 960 -> 1280)
MOST_BYTES = 3.7e9
MOST_FLOPS = 4.0e12


def listed():
    return [
        # One image through all 34 pointwise layers: interactive inference, where latency counts.
        {"name": "sequence_b1", "kind": "sequence", "batch": 1, "h0": 112, "width": 1.0, "depthwise": False},
        # The benchmark's workload: the same layers at batch 128.
        {"name": "sequence_b128", "kind": "sequence", "batch": 128, "h0": 112, "width": 1.0, "depthwise": False},
        # The network body as it is deployed: depthwise 3x3 layers, linear project layers, skip connections.
        {"name": "body_b64", "kind": "sequence", "batch": 64, "h0": 112, "width": 1.0, "depthwise": True},
        # The body at width 0.75 and an odd batch: channel counts that are 8 modulo 16, odd row counts.
        {"name": "body_b9_w075", "kind": "sequence", "batch": 9, "h0": 112, "width": 0.75, "depthwise": True},
        # One small layer (batch 1, 14 x 14): the cost of a call.
        {"name": "conv_196x64x384", "kind": "conv", "m": 196, "cin": 64, "cout": 384, "option": "plain"},
        # An early expand layer, batch 64 at 112 x 112: bound by its bytes.
        {"name": "conv_802816x16x96", "kind": "conv", "m": 802816, "cin": 16, "cout": 96, "option": "plain"},
        # The heaviest contraction of the shape sweep.
        {"name": "conv_1605632x960x1280", "kind": "conv", "m": 1605632, "cin": 960, "cout": 1280, "option": "plain"},
        # The head layer at batch 512 from operands prepared ahead of the call: a server's steady state.
        {"name": "prepared_25088x320x1280", "kind": "conv", "m": 25088, "cin": 320, "cout": 1280, "option": "prepared"},
        # The paper's own dataflow: a layer that dequantises and re-quantises per sample.
        {"name": "dynamic_b128_16x96", "kind": "dynamic", "batch": 128, "rows": 12544, "cin": 16, "cout": 96},
        # Its activation quantiser, on the stem's output at batch 128.
        {"name": "act_b128_112x112x32", "kind": "act", "batch": 128, "h": 112, "w": 112, "c": 32},
        # A depthwise layer on its own, with stride 2 (the body has both strides at every size).
        {"name": "depthwise_b128_112x96_s2", "kind": "depthwise", "batch": 128, "h": 112, "w": 112, "c": 96, "stride": 2},
        # Float weights of the whole network to 2-bit codes: once per model load or training step.
        {"name": "weights_w10", "kind": "weights", "width": 1.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_once(rng):
    kind = rng.choice(("sequence", "body", "conv", "conv", "prepared", "dynamic", "act", "depthwise", "weights"))
    if kind in ("sequence", "body"):
        return {"kind": "sequence", "batch": _log_int(rng, 1, 160), "h0": rng.choice((64, 80, 96, 112)),
                "width": rng.choice(WIDTHS), "depthwise": kind == "body"}
    if kind in ("conv", "prepared"):
        cin, cout = rng.choice(NARROW), rng.choice(WIDE)
        if rng.random() < 0.5:
            cin, cout = cout, cin
        if kind == "conv" and rng.random() < 0.15:
            cin, cout = rng.choice((512, 768, 960)), rng.choice((320, 512, 1280))
        side = rng.choice(SPATIAL)
        m = _log_int(rng, 1, max(1, 1605632 // (side * side))) * side * side
        option = "prepared" if kind == "prepared" else rng.choice(("plain", "plain", "linear", "residual"))
        if option == "prepared" and (cin % 16 or cout % 16):
            m += m % 2          # the prepared form takes such channel counts on even row counts only
        return {"kind": "conv", "m": m, "cin": cin, "cout": cout, "option": option}
    if kind == "dynamic":
        side = rng.choice(SPATIAL)
        return {"kind": "dynamic", "batch": _log_int(rng, 1, 160), "rows": side * side,
                "cin": rng.choice([c for c in NARROW + WIDE if c % 16 == 0]),
                "cout": rng.choice([c for c in NARROW + WIDE if c % 16 == 0 or (c % 8 == 0 and c <= 256)])}
    if kind == "act":
        side = rng.choice(SPATIAL)
        return {"kind": "act", "batch": _log_int(rng, 1, 192), "h": side, "w": side, "c": rng.choice(NARROW + WIDE)}
    if kind == "depthwise":
        side = rng.choice(SPATIAL)
        return {"kind": "depthwise", "batch": _log_int(rng, 1, 192), "h": side, "w": side,
                "c": rng.choice(NARROW + WIDE), "stride": rng.choice((1, 2))}
    return {"kind": "weights", "width": round(rng.uniform(0.5, 2.0), 2)}


def draw(rng):
    while True:
        case = _draw_once(rng)
        w = work(case)
        if w["bytes"] <= MOST_BYTES and w["flops"] <= MOST_FLOPS:
            return case


# ---- shapes -------------------------------------------------------------------------------------

def _layers(case):
    return synth.mobilenetv2_pointwise_layers(h0=case["h0"], w0=case["h0"], width=case["width"])


def _has_depthwise(case, layer):
    return case["depthwise"] and layer.name.endswith("project")


def work(case):
    kind = case["kind"]
    if kind == "sequence":
        layers, b, nbytes, flops = _layers(case), case["batch"], 0, 0
        for i, l in enumerate(layers):
            m = b * l.h * l.w
            nbytes += m * (l.cin + l.cout) + l.cout * l.cin // 4 + 9 * l.cout
            flops += 2 * m * l.cin * l.cout
            if _has_depthwise(case, l):
                nbytes += b * (l.h * l.in_stride) * (l.w * l.in_stride) * l.cin + m * l.cin + 18 * l.cin
                flops += 2 * 9 * m * l.cin
                if synth.has_skip_connection(layers, i):
                    nbytes += m * l.cout
        return {"bytes": nbytes, "flops": flops}
    if kind == "conv":
        m, k, n = case["m"], case["cin"], case["cout"]
        out = 2 if case["option"] == "residual" else 1
        return {"bytes": m * (k + out * n) + n * k // 4 + 9 * n, "flops": 2 * m * k * n}
    if kind == "dynamic":
        m, k, n = case["batch"] * case["rows"], case["cin"], case["cout"]
        return {"bytes": m * (k + n) + n * k // 4 + 4 * n + 12 * case["batch"], "flops": 2 * m * k * n}
    if kind == "act":
        n = case["batch"] * case["h"] * case["w"] * case["c"]
        return {"bytes": 5 * n + 8 * case["batch"], "flops": 3 * n}
    if kind == "depthwise":
        b, h, w, c, s = (case[k] for k in ("batch", "h", "w", "c", "stride"))
        out = b * ((h - 1) // s + 1) * ((w - 1) // s + 1) * c
        return {"bytes": b * h * w * c + out + 18 * c, "flops": 18 * out}
    weights = [(l.cout, l.cin) for l in synth.mobilenetv2_pointwise_layers(width=case["width"])]
    return {"bytes": sum(4 * n * k + n * ((k + 3) // 4) + 4 * n for n, k in weights),
            "flops": sum(3 * n * k for n, k in weights)}


def tolerance(case):
    # Integer sums, fixed-point rounding and the quantisers' single binary32 operations have one
    # correct result.  Only the weight quantiser returns a float that depends on the order of a sum
    # (taken in binary64, returned as binary32).
    return {"rel": 1e-6, "differ": 0.0} if case["kind"] == "weights" else "exact"


# ---- inputs -------------------------------------------------------------------------------------

class _Source:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda")
        self.g.manual_seed(seed)

    def ints(self, lo, hi, shape, dtype):
        return torch.randint(lo, hi, shape, generator=self.g, device="cuda", dtype=dtype)

    def normal(self, shape):
        return torch.randn(shape, generator=self.g, device="cuda")

    def activations(self, shape, signed=False):
        """Post-ReLU6 int8 values, or symmetric ones."""
        if signed:
            return self.ints(-127, 128, shape, torch.int8)
        # three tenths of [-54, 127] lie below zero and are clamped to it
        return self.ints(-54, 128, shape, torch.int8).clamp_(min=0)

    def ternary(self, cout, cin):
        # the difference of two bits: P(0) = 1/2, P(+1) = P(-1) = 1/4
        return self.ints(0, 2, (cout, cin), torch.int8) - self.ints(0, 2, (cout, cin), torch.int8)

    def requant(self, cout, fan_in, rms_in, rms_out=45.0):
        """(bias, mult, shift): accumulators of `fan_in` products with half of the weights zero go to
        about `rms_out`; the scales of the channels span a factor of eight."""
        acc = math.sqrt(fan_in / 2.0) * rms_in
        shift = max(0, int(math.floor(math.log2(acc / rms_out))) - 1) + self.ints(0, 3, (cout,), torch.int32)
        bias = self.ints(-int(acc / 2) - 1, int(acc / 2) + 2, (cout,), torch.int32)
        return bias, self.ints(1 << 30, (1 << 31) - 1, (cout,), torch.int32), shift.to(torch.int8)


def _prepare_sequence(case, src):
    shapes, layers, signed = _layers(case), [], False
    for i, l in enumerate(shapes):
        bias, mult, shift = src.requant(l.cout, l.cin, 60.0)
        d = dict(cin=l.cin, cout=l.cout, in_stride=l.in_stride, bias=bias, mult=mult, shift=shift,
                 w_packed=binding.pack_ternary(src.ternary(l.cout, l.cin)))
        if _has_depthwise(case, l):
            # project layers are linear and carry the block's skip connection; 8-bit depthwise filters
            d["dw_w"] = src.ints(-127, 128, (l.cin, 3, 3), torch.int8)
            db, dm, ds = src.requant(l.cin, 18, 60.0 * 73.0)
            d.update(dw_bias=db, dw_mult=dm, dw_shift=ds, act_min=-128,
                     add_block_input=synth.has_skip_connection(shapes, i))
        layers.append(d)
    seq = binding.LayerSeq(layers)
    b, h0 = case["batch"], case["h0"]
    ws = torch.empty(seq.workspace_bytes(b, h0, h0), dtype=torch.uint8, device="cuda")
    side = h0 // seq.total_stride
    return dict(seq=seq, x=src.activations((b, h0, h0, shapes[0].cin)), ws=ws,
                y=torch.empty((b, side, side, seq.cout_last), dtype=torch.int8, device="cuda"))


def _prepare_conv(case, src):
    m, k, n, option = case["m"], case["cin"], case["cout"], case["option"]
    lo = -128 if option in ("linear", "residual") else 0
    rq = binding.make_requant(*src.requant(n, k, 60.0), lo, 127)
    s = dict(rq=rq, wp=binding.pack_ternary(src.ternary(n, k)), x=src.activations((m, k)),
             y=torch.empty((m, n), dtype=torch.int8, device="cuda"))
    if option == "prepared":
        s["operands"] = binding.pw_prepare(m, k, s["wp"], n, rq)
    if option == "residual":
        s["res"] = src.activations((m, n), signed=True)
    return s


def prepare(case, seed):
    src, kind = _Source(seed), case["kind"]
    if kind == "sequence":
        s = _prepare_sequence(case, src)
    elif kind == "conv":
        s = _prepare_conv(case, src)
    elif kind == "dynamic":
        b, rows, k, n = case["batch"], case["rows"], case["cin"], case["cout"]
        x = src.activations((b * rows, k), signed=True)
        s = dict(x=x, wp=binding.pack_ternary(src.ternary(n, k)),
                 alpha=src.normal((n,)).abs_().mul_(0.02).add_(0.03), gamma=src.normal((b,)).abs_().add_(3.0),
                 out=(torch.empty((b * rows, n), dtype=torch.int8, device="cuda"),
                      torch.empty((b,), device="cuda"), torch.empty((b,), device="cuda")))
    elif kind == "act":
        x = src.normal((case["batch"], case["h"], case["w"], case["c"]))
        b = case["batch"]
        s = dict(x=x, out=(torch.empty(x.shape, dtype=torch.int8, device="cuda"),
                           torch.empty((b,), device="cuda"), torch.empty((b,), device="cuda")))
    elif kind == "depthwise":
        b, h, w, c, stride = (case[k] for k in ("batch", "h", "w", "c", "stride"))
        s = dict(x=src.activations((b, h, w, c)), w=src.ints(-127, 128, (c, 3, 3), torch.int8),
                 rq=binding.make_requant(*src.requant(c, 18, 60.0 * 73.0)),
                 y=torch.empty((b, (h - 1) // stride + 1, (w - 1) // stride + 1, c), dtype=torch.int8, device="cuda"))
    else:
        shapes = synth.mobilenetv2_pointwise_layers(width=case["width"])
        s = dict(jobs=binding.QuantizeJobs([src.normal((l.cout, l.cin)).mul_(math.sqrt(2.0 / l.cin)) for l in shapes]))
    s["case"] = case
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "sequence":
        return binding.pw_layer_seq(state["seq"], state["x"], state["ws"], state["y"])
    if kind == "conv":
        if case["option"] == "prepared":
            return binding.pw_conv_i8_prepared(state["x"], case["cout"], state["operands"], y=state["y"])
        if case["option"] == "residual":
            return binding.pw_conv_i8_res(state["x"], state["wp"], case["cout"], state["rq"], state["res"], y=state["y"])
        return binding.pw_conv_i8(state["x"], state["wp"], case["cout"], state["rq"], y=state["y"])
    if kind == "dynamic":
        return binding.pw_conv_i8_dyn(state["x"], case["batch"], state["wp"], case["cout"], state["alpha"],
                                      state["gamma"], out=state["out"])
    if kind == "act":
        return binding.quantize_act_absmax(state["x"], out=state["out"])
    if kind == "depthwise":
        return binding.dw_conv3x3_i8(state["x"], state["w"], state["rq"], stride=case["stride"], y=state["y"])
    # 34 matrices: the codes and the scales of all of them
    packed = binding.quantize_ternary_batch(jobs=state["jobs"])
    return {"packed": [p for p, _ in packed][:32], "alpha": [a for _, a in packed][:32]}
