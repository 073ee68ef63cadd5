"""The work that users of this library have it do, as cases that can be timed and compared.

A case is a dict of plain values; ``prepare`` makes what a user's program holds before the call
(device tensors with the value recipe of the repository's benchmark, epilogue constants, output
buffers), ``run`` makes one pass through the public entry points, ``work`` says what that pass
cannot do without.

Kinds: ``gemm`` and ``conv`` (one fused layer), ``net`` (the bottleneck stack of ResNet-50,
chained, with its residual inputs), ``transform`` (the standalone activation transform),
``codec`` (packed stream, encode and decode), ``calibrate`` (min-max front end) and ``sparse24``
(a GEMM on 2:4 pruned weights).
"""
from __future__ import annotations

import math

import torch

import paper_2105_11010_b200 as sparq

# mode, window bits, placement set, rounding
VARIANTS = {
    "vsparq-5opt": (sparq.MODE_VSPARQ, 4, sparq.SET_5OPT, sparq.ROUND_NEAREST),
    "vsparq-5opt-trim": (sparq.MODE_VSPARQ, 4, sparq.SET_5OPT, sparq.ROUND_TRUNCATE),
    "vsparq-3opt": (sparq.MODE_VSPARQ, 4, sparq.SET_3OPT, sparq.ROUND_NEAREST),
    "vsparq-2opt": (sparq.MODE_VSPARQ, 4, sparq.SET_2OPT, sparq.ROUND_NEAREST),
    "bsparq-5opt": (sparq.MODE_BSPARQ, 4, sparq.SET_5OPT, sparq.ROUND_NEAREST),
    "vsparq-6opt": (sparq.MODE_VSPARQ, 3, sparq.SET_6OPT, sparq.ROUND_NEAREST),
    "vsparq-7opt": (sparq.MODE_VSPARQ, 2, sparq.SET_7OPT, sparq.ROUND_NEAREST),
    "none": (sparq.MODE_NONE, 4, sparq.SET_5OPT, sparq.ROUND_NEAREST),
}


def listed():
    return [
        # One small layer: a 256-row GEMM with int32 and fp32 outputs (the library's smallest
        # benchmark config). Launches and latency.
        {"name": "gemm-256x64x576", "kind": "gemm", "m": 256, "n": 64, "k": 576, "variant": "vsparq-5opt",
         "outputs": "acc+f32"},
        # A large fully connected layer: compute-bound GEMM, requantized bytes out.
        {"name": "gemm-16384x4096x4096", "kind": "gemm", "m": 16384, "n": 4096, "k": 4096, "variant": "vsparq-5opt",
         "outputs": "u8"},
        # ResNet-18-style 3x3 layer at batch 32.
        {"name": "conv-32x56x56x64", "kind": "conv", "batch": 32, "h": 56, "w": 56, "c": 64, "cout": 64, "r": 3,
         "stride": 1, "pad": 1, "variant": "vsparq-5opt", "outputs": "u8"},
        # The ablation layer: 3x3, 128 channels, batch 128 (the benchmark's headline).
        {"name": "conv-128x28x28x128", "kind": "conv", "batch": 128, "h": 28, "w": 28, "c": 128, "cout": 128, "r": 3,
         "stride": 1, "pad": 1, "variant": "vsparq-5opt", "outputs": "u8"},
        # An inception-style 5x5 branch: odd batch and image size, 48 channels (not a whole
        # reduction block), a restricted placement set, dequantized fp32 out.
        {"name": "conv-17x35x35x48-5x5", "kind": "conv", "batch": 17, "h": 35, "w": 35, "c": 48, "cout": 64, "r": 5,
         "stride": 1, "pad": 2, "variant": "vsparq-3opt", "outputs": "f32"},
        # Inference of the whole bottleneck stack: throughput (batch 64) and latency (one image).
        {"name": "resnet50-batch64", "kind": "net", "batch": 64, "variant": "vsparq-5opt"},
        {"name": "resnet50-batch1", "kind": "net", "batch": 1, "variant": "vsparq-5opt"},
        # The standalone transform on 2^30 activations.
        {"name": "transform-2p30", "kind": "transform", "rows": 1 << 20, "row_len": 1024, "variant": "vsparq-5opt"},
        # Activations stored in packed form between layers: encode, then decode (the 4-bit form
        # and the 3-bit one).
        {"name": "codec-5opt", "kind": "codec", "rows": 200704, "row_len": 256, "variant": "vsparq-5opt"},
        {"name": "codec-6opt", "kind": "codec", "rows": 200704, "row_len": 256, "variant": "vsparq-6opt"},
        # Post-training quantization of one layer: statistics and u8 activations of a calibration
        # batch (bf16), s8 weights.
        {"name": "calibrate-bf16", "kind": "calibrate", "n": 64 * 56 * 56 * 256, "dtype": "bf16", "cout": 512,
         "k": 4608},
        # The 3x3 layer of the 28x28x128 maps as a GEMM with 2:4 pruned weights.
        {"name": "sparse24-100352x128x1152", "kind": "sparse24", "m": 100352, "n": 128, "k": 1152,
         "variant": "vsparq-5opt"},
    ]


def _log(rng, lo, hi):
    """An integer of [lo, hi], spread over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["gemm", "conv", "net", "transform", "codec", "calibrate", "sparse24"])
    v = rng.choice(sorted(VARIANTS))
    spar = rng.choice(sorted(k for k in VARIANTS if k != "none"))
    if kind == "gemm":
        return {"kind": kind, "m": _log(rng, 64, 16384), "n": _log(rng, 4, 512) * 8 - rng.choice([0, 0, 0, 3]),
                "k": _log(rng, 4, 256) * 16, "variant": v, "outputs": rng.choice(["u8", "u8", "f32", "acc+f32"])}
    if kind == "conv":
        while True:
            hw, r = rng.choice([7, 14, 28, 56, rng.randint(7, 56)]), rng.choice([1, 3, 3, 5])
            c = {"kind": kind, "batch": _log(rng, 1, 128), "h": hw, "w": hw, "c": _log(rng, 1, 32) * 16,
                 "cout": _log(rng, 2, 64) * 8, "r": r, "stride": rng.choice([1, 1, 1, 2]), "pad": r // 2,
                 "variant": v, "outputs": rng.choice(["u8", "u8", "f32"])}
            w = work(c)
            if w["flops"] <= 1e11 and w["bytes"] <= 4e8:
                return c
    if kind == "net":
        return {"kind": kind, "batch": _log(rng, 1, 64), "variant": v}
    if kind == "transform":
        row = rng.choice([64, 256, 1024, 4608, rng.randint(50, 3000)])
        return {"kind": kind, "rows": max(1, _log(rng, 1 << 12, 1 << 30) // row), "row_len": row, "variant": v}
    if kind == "codec":
        row = rng.randint(2, 64) * 16
        return {"kind": kind, "rows": max(1, _log(rng, 1 << 14, 1 << 26) // row), "row_len": row, "variant": spar}
    if kind == "calibrate":
        return {"kind": kind, "n": _log(rng, 1 << 14, 1 << 26), "dtype": rng.choice(["bf16", "f32"]),
                "cout": _log(rng, 16, 2048), "k": _log(rng, 4, 288) * 16}
    return {"kind": kind, "m": _log(rng, 49, 100352), "n": _log(rng, 4, 64) * 8, "k": _log(rng, 4, 72) * 16,
            "variant": spar}


# ---- inputs ---------------------------------------------------------------------------------

def _activations(g, count, zero_frac=0.5):
    """uint8: zeros with probability ``zero_frac``, else clip(round(|N(0,1)| * 40), 1, 255)."""
    out = torch.empty(count, dtype=torch.uint8, device="cuda")
    for lo in range(0, count, 1 << 26):
        part = out[lo:lo + (1 << 26)]
        z = torch.randn(part.numel(), generator=g, device="cuda")
        v = z.abs_().mul_(40.0).round_().clamp_(1, 255).to(torch.uint8)
        v[torch.rand(part.numel(), generator=g, device="cuda") < zero_frac] = 0
        part.copy_(v)
    return out


def _weights(g, *shape):
    """int8: clip(round(N(0,1) * 30), -127, 127)."""
    return (torch.randn(shape, generator=g, device="cuda") * 30.0).round_().clamp_(-127, 127).to(torch.int8)


def _constants(g, cout):
    scale = 0.001 + 0.009 * torch.rand(cout, generator=g, device="cuda")
    bias = 2.0 * torch.rand(cout, generator=g, device="cuda") - 1.0
    return scale, bias


def _inv_out_scale(k):
    """One standard deviation of the dequantized output lands on 40 of the next layer's u8 grid."""
    return 40.0 / (math.sqrt(k * 0.5 * 1600.0 * 900.0) * 0.0055)


def _outputs(kind, shape):
    new = lambda dt: torch.empty(shape, dtype=dt, device="cuda")  # noqa: E731
    return {"acc+f32": lambda: {"acc_out": new(torch.int32), "f32_out": new(torch.float32)},
            "f32": lambda: {"f32_out": new(torch.float32)},
            "u8": lambda: {"u8_out": new(torch.uint8)}}[kind]()


def _layer(g, batch, h, w, c, cout, r, stride, pad, outputs="u8", relu=True):
    """One convolution's resident data and its output buffers."""
    ho, wo = (h + 2 * pad - r) // stride + 1, (w + 2 * pad - r) // stride + 1
    scale, bias = _constants(g, cout)
    return {"w": _weights(g, cout, r, r, c), "stride": (stride, stride), "pad": (pad, pad),
            "args": dict(scale=scale, bias=bias, relu=relu, inv_out_scale=_inv_out_scale(r * r * c),
                         **_outputs(outputs, (batch, ho, wo, cout)))}


def _blocks():
    """The 16 bottleneck blocks of ResNet-50: (map size, channels in, middle, stride, has projection)."""
    hw, cin, out = 56, 64, []
    for stage, (mid, count) in enumerate([(64, 3), (128, 4), (256, 6), (512, 3)]):
        for b in range(count):
            stride = 2 if (b == 0 and stage > 0) else 1
            out.append((hw, cin, mid, stride, b == 0))
            hw, cin = hw // stride, 4 * mid
    return out


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    kind = case["kind"]
    params = sparq.SparqParams(*VARIANTS[case["variant"]]) if "variant" in case else None
    s = {"kind": kind, "params": params}
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        scale, bias = _constants(g, n)
        s.update(a=_activations(g, m * k).view(m, k), b=_weights(g, n, k),
                 args=dict(scale=scale, bias=bias, relu=case["outputs"] == "u8", inv_out_scale=_inv_out_scale(k),
                           **_outputs(case["outputs"], (m, n))))
    elif kind == "conv":
        nb, h, c = case["batch"], case["h"], case["c"]
        s.update(x=_activations(g, nb * h * case["w"] * c).view(nb, h, case["w"], c),
                 layer=_layer(g, nb, h, case["w"], c, case["cout"], case["r"], case["stride"], case["pad"],
                              case["outputs"]))
    elif kind == "net":
        nb = case["batch"]
        s.update(x=_activations(g, nb * 56 * 56 * 64).view(nb, 56, 56, 64), blocks=[])
        for hw, cin, mid, stride, proj in _blocks():
            ho = hw // stride
            block = {"a": _layer(g, nb, hw, hw, cin, mid, 1, 1, 0), "b": _layer(g, nb, hw, hw, mid, mid, 3, stride, 1),
                     "c": _layer(g, nb, ho, ho, mid, 4 * mid, 1, 1, 0)}
            if proj:
                block["p"] = _layer(g, nb, hw, hw, cin, 4 * mid, 1, stride, 0, relu=False)
            # the identity tensor's own scale: half a standard deviation of the block's sum
            block["residual_scale"] = 0.5 / block["c"]["args"]["inv_out_scale"]
            s["blocks"].append(block)
    elif kind == "transform":
        s.update(rows=case["rows"], row_len=case["row_len"], x=_activations(g, case["rows"] * case["row_len"]))
        s["y"] = torch.empty_like(s["x"])
    elif kind == "codec":
        count = case["rows"] * case["row_len"]
        s["x"] = _activations(g, count).view(case["rows"], case["row_len"])
        s["data"] = torch.empty(count // 16 * 2 * params.window_bits, dtype=torch.uint8, device="cuda")
        s["ctrl"] = torch.empty(count // 16 * sparq.sparq_packed_ctrl_bits(params), dtype=torch.uint8, device="cuda")
        s["y"] = torch.empty_like(s["x"])
    elif kind == "calibrate":
        dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
        x = torch.empty(case["n"], dtype=dt, device="cuda")
        for lo in range(0, case["n"], 1 << 26):        # post-ReLU activations
            part = x[lo:lo + (1 << 26)]
            part.copy_(torch.randn(part.numel(), generator=g, device="cuda").clamp_(min=0.0))
        s.update(x=x, w=torch.randn((case["cout"], case["k"]), generator=g, device="cuda") * 0.05,
                 max=torch.zeros(1, device="cuda"), q=torch.empty(case["n"], dtype=torch.uint8, device="cuda"),
                 wq=torch.empty((case["cout"], case["k"]), dtype=torch.int8, device="cuda"),
                 ws=torch.empty(case["cout"], device="cuda"))
    else:
        m, n, k = case["m"], case["n"], case["k"]
        patterns = torch.tensor([(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)], dtype=torch.uint8, device="cuda")
        pos = patterns[torch.randint(0, 6, (n, k // 4), generator=g, device="cuda")].view(n, k // 2).contiguous()
        kx = sparq.sparq_sparse24_expanded_k(k, params)
        w_exp = torch.empty((n, kx), dtype=torch.int8, device="cuda")
        sparq.sparq_sparse24_expand_weights(_weights(g, n, k // 2), pos, params, w_exp)
        scale, bias = _constants(g, n)
        s.update(a=_activations(g, m * k).view(m, k), w=w_exp,
                 args=dict(workspace=torch.empty(m * kx, dtype=torch.uint8, device="cuda"), scale=scale, bias=bias,
                           relu=True, inv_out_scale=_inv_out_scale(k // 2), **_outputs("u8", (m, n))))
    return s


# ---- one pass ----------------------------------------------------------------------------------

def _conv(x, layer, params, **more):
    sparq.sparq_conv2d_nhwc_s8(x, layer["w"], layer["stride"], layer["pad"], params, **layer["args"], **more)
    return layer["args"]["u8_out"]


def run(s):
    kind, params = s["kind"], s["params"]
    if kind == "gemm":
        sparq.sparq_gemm_s8(s["a"], s["b"], params, **s["args"])
        return [v for k, v in s["args"].items() if k.endswith("_out")]
    if kind == "conv":
        layer = s["layer"]
        sparq.sparq_conv2d_nhwc_s8(s["x"], layer["w"], layer["stride"], layer["pad"], params, **layer["args"])
        return [v for k, v in layer["args"].items() if k.endswith("_out")]
    if kind == "net":
        x, outs = s["x"], []
        for b in s["blocks"]:
            identity = _conv(x, b["p"], params) if "p" in b else x
            x = _conv(_conv(_conv(x, b["a"], params), b["b"], params), b["c"], params, residual=identity,
                      residual_scale=b["residual_scale"])
            outs.append(x)
        return outs
    if kind == "transform":
        sparq.sparq_quantize(s["x"], s["y"], s["rows"], s["row_len"], params)
        return s["y"]
    if kind == "codec":
        sparq.sparq_pack(s["x"], params, s["data"], s["ctrl"])
        sparq.sparq_unpack(s["data"], s["ctrl"], params, s["y"])
        return [s["data"], s["ctrl"], s["y"]]
    if kind == "calibrate":
        s["max"].zero_()
        sparq.sparq_absmax(s["x"], s["max"])
        sparq.sparq_quantize_act_u8(s["x"], s["max"], s["q"])
        sparq.sparq_quantize_weight_s8(s["w"], s["wq"], s["ws"])
        return [s["max"], s["q"], s["wq"], s["ws"]]
    sparq.sparq_gemm_s8_sparse24(s["a"], s["w"], params, **s["args"])
    return s["args"]["u8_out"]


# ---- what a pass cannot do without ------------------------------------------------------------

OUT_BYTES = {"u8": 1, "f32": 4, "acc+f32": 8}


def _conv_work(batch, h, w, c, cout, r, stride, pad, out_bytes=1, residual=False):
    m = batch * ((h + 2 * pad - r) // stride + 1) * ((w + 2 * pad - r) // stride + 1)
    # a strided 1x1 filter never reads the pixels between its taps
    read = m * c if r == 1 else batch * h * w * c
    return (read + cout * r * r * c + 8 * cout + m * cout * (out_bytes + (1 if residual else 0)),
            2.0 * m * cout * r * r * c)


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": m * k + n * k + 8 * n + m * n * OUT_BYTES[case["outputs"]], "flops": 2.0 * m * n * k}
    if kind == "conv":
        b, f = _conv_work(case["batch"], case["h"], case["w"], case["c"], case["cout"], case["r"], case["stride"],
                          case["pad"], OUT_BYTES[case["outputs"]])
        return {"bytes": b, "flops": f}
    if kind == "net":       # every layer reads its input and writes its output
        parts = []
        for hw, cin, mid, stride, proj in _blocks():
            ho = hw // stride
            parts += [_conv_work(case["batch"], hw, hw, cin, mid, 1, 1, 0),
                      _conv_work(case["batch"], hw, hw, mid, mid, 3, stride, 1),
                      _conv_work(case["batch"], ho, ho, mid, 4 * mid, 1, 1, 0, residual=True)]
            if proj:
                parts.append(_conv_work(case["batch"], hw, hw, cin, 4 * mid, 1, stride, 0))
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "transform":
        return {"bytes": 2 * case["rows"] * case["row_len"], "flops": 0}
    if kind == "codec":     # encode: activations in, planes out; decode: planes in, activations out
        count = case["rows"] * case["row_len"]
        p = sparq.SparqParams(*VARIANTS[case["variant"]])
        planes = count // 16 * (2 * p.window_bits + sparq.sparq_packed_ctrl_bits(p))
        return {"bytes": 2 * (count + planes), "flops": 0}
    if kind == "calibrate":
        # the maximum has to be known before the first byte is quantized: x is read twice
        width = 2 if case["dtype"] == "bf16" else 4
        return {"bytes": case["n"] * (2 * width + 1) + case["cout"] * (case["k"] * 5 + 4), "flops": 0}
    m, n, k = case["m"], case["n"], case["k"]       # half of the weights are zeros; K/2 values and coordinates
    return {"bytes": m * k + n * k + 8 * n + m * n, "flops": 1.0 * m * n * k}


def tolerance(case):
    # Bytes and accumulators are exact; the fp32 outputs are one fused multiply-add of an exact
    # integer, so another correct implementation differs by rounding at most.
    return {"rel": 1e-6, "max": 1e-5} if "f32" in case.get("outputs", "") else "exact"
