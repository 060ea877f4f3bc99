"""Workloads of the GDWS forward whose time matters to a user, through the library's public entry points.

A case is a dict of plain values: `kind` says which entry points a pass takes, the rest is the layer's shape and options.

    forward   one Plan.forward with weights packed beforehand (bf16) or read in place (fp32): inference on a loaded network
    weights   one Plan.forward that is given the weights with the call: weights that change from call to call
    chain     the 16 residual-block 3x3 layers of a CIFAR ResNet-18, ReLU between them, one Plan.forward per layer
    stages    Plan.depthwise, then Plan.pointwise: the two convolutions as separate calls, z in a buffer of the caller's
    host      Plan.forward_host: activations in pinned host memory, copied in and out by the call

Shapes and value distributions follow `paper_2110_14871_b200.inputs` (layers of the paper's CIFAR and ImageNet networks).
The multipliers g_c belong to the network and are drawn from the case's sizes; activations and weights come from the seed.
"""
import math

import numpy as np
import torch

from paper_2110_14871_b200 import gdws
from paper_2110_14871_b200 import inputs as gi


def _layer(name, kind, n, c, d, h, w, g, k=3, stride=1, dtype="bf16", layout="NHWC", relu=False, out_f32=False):
    """g: "heavy", or "lo-hi" for uniform multipliers."""
    case = {"kind": kind, "n": n, "c": c, "d": d, "h": h, "w": w, "k": k, "stride": stride, "g": g, "dtype": dtype,
            "layout": layout, "relu": relu, "out_f32": out_f32}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the smallest call: one small fp32 image (launch and call overhead count)
        _layer("f32_small", "forward", 1, 16, 16, 32, 32, "1-3", dtype="f32", layout="NCHW"),
        # fp32 at an ordinary batch of a CIFAR / ImageNet middle layer
        _layer("f32_batch", "forward", 16, 128, 128, 28, 28, "1-9", dtype="f32", layout="NCHW"),
        # one image at a time through a ResNet-50 middle layer: interactive inference
        _layer("one_image", "forward", 1, 256, 256, 14, 14, "heavy"),
        # VGG-16 middle layer on CIFAR images, the library's default benchmark
        _layer("vgg_cifar", "forward", 256, 256, 256, 8, 8, "1-9"),
        # ResNet-50 layer that halves the resolution
        _layer("resnet50_stride2", "forward", 64, 128, 128, 56, 56, "heavy", stride=2),
        # odd batch, odd map, channel counts off the powers of two, fp32 sums kept, weights new on each call
        _layer("ragged_weights", "weights", 37, 72, 120, 45, 51, "heavy", relu=True, out_f32=True),
        # 16 layers in a row, ReLU between them: batch inference of CIFAR images
        {"name": "resnet18_chain", "kind": "chain", "n": 512, "c": 64, "h": 32, "w": 32, "g": "1-9"},
        # first 3x3 layer of VGG-16 on ImageNet images: the largest activations
        _layer("vgg_first", "forward", 32, 64, 64, 224, 224, "heavy"),
        # a wide VGG-16 layer: the pointwise part dominates
        _layer("vgg_wide", "forward", 32, 512, 512, 28, 28, "heavy"),
        # 5x5 filters: the most arithmetic
        _layer("five_by_five", "forward", 32, 256, 256, 56, 56, "1-25", k=5),
        # the two stages on their own
        _layer("stages", "stages", 64, 64, 64, 56, 56, "heavy"),
        # activations on the host
        _layer("host_buffers", "host", 256, 256, 256, 8, 8, "1-9"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# A drawn layer is kept within these: multiply-adds of the bf16 and fp32 layers, elements of one activation tensor.
_MAX_MACS_BF16, _MAX_MACS_F32, _MAX_ELEMS = 8e10, 1.2e9, 1e8


def draw(rng):
    kind = rng.choices(["forward", "f32", "weights", "chain", "stages", "host"], [10, 3, 2, 1, 2, 2])[0]
    if kind == "chain":
        return {"kind": "chain", "n": int(_log(rng, 8, 400)), "c": rng.choice([32, 48, 64]), "h": rng.randint(24, 36),
                "w": rng.randint(24, 36), "g": rng.choice(["1-9", "heavy"])}
    f32 = kind == "f32"
    while True:
        k = rng.choice([3, 3, 3, 3, 5])
        stride = rng.choice([1, 1, 1, 2])
        if f32:
            c, d = int(_log(rng, 8, 256)), int(_log(rng, 8, 256))
        else:
            c, d = (8 * int(round(_log(rng, 16, 512) / 8)) for _ in range(2))
        h = max(5, int(_log(rng, 6, 224)))
        w = max(5, min(224, int(h * rng.uniform(0.7, 1.4))))
        n = int(_log(rng, 1, 257))
        g = rng.choice(["heavy", "1-9", "1-3"]) if k == 3 else rng.choice(["heavy", "1-25"])
        case = _layer(None, "forward" if f32 else kind, n, c, d, h, w, g, k, stride, "f32" if f32 else "bf16",
                      rng.choice(["NCHW", "NHWC"]) if f32 else "NHWC", rng.random() < 0.5,
                      kind in ("forward", "weights") and rng.random() < 0.15)
        s = _spec(case)
        elems = max(n * h * w * c, n * s.Ho * s.Wo * d)
        macs = n * s.Ho * s.Wo * int(_g(case).sum()) * (k * k + d)
        most = 2e7 if kind in ("stages", "host") else _MAX_ELEMS
        if elems <= most and macs <= (_MAX_MACS_F32 if f32 else _MAX_MACS_BF16):
            return case


def _layers(case):
    """The case's layers as single-layer cases."""
    if case["kind"] != "chain":
        return [case]
    out, cin, h, w = [], case["c"], case["h"], case["w"]
    for stage in range(4):
        width = case["c"] << stage
        for block in range(4):
            stride = 2 if stage > 0 and block == 0 else 1
            out.append(_layer(None, "forward", case["n"], cin, width, h, w, case["g"], 3, stride, relu=len(out) < 15))
            h, w, cin = gi.out_dim(h, 3, stride, 1), gi.out_dim(w, 3, stride, 1), width
    return out


def _g(layer):
    dist = ("heavy",) if layer["g"] == "heavy" else ("uniform",) + tuple(int(v) for v in layer["g"].split("-"))
    key = [layer[k] for k in ("n", "c", "d", "h", "w", "k", "stride")]
    return gi.make_g(np.random.Generator(np.random.PCG64(key)), layer["c"], dist)


def _spec(layer):
    return gi.LayerSpec("layer", layer["n"], layer["c"], layer["d"], layer["h"], layer["w"], layer["k"], layer["stride"],
                        layer["k"] // 2, dtype=layer["dtype"], layout=layer["layout"])


def _shape(layout, n, c, h, w):
    return (n, c, h, w) if layout == "NCHW" else (n, h, w, c)


def _prepare_layer(layer, gen, with_x=True):
    s = _spec(layer)
    f32 = layer["dtype"] == "f32"
    dtype = torch.float32 if f32 else torch.bfloat16
    g = _g(layer)
    G = int(g.sum())

    def normal(shape, sd):
        return (torch.randn(shape, generator=gen, device="cuda") * sd).to(dtype)

    plan = gdws.Plan(s.C, s.D, s.k, s.stride, s.pad, g)
    plan.set_option(gdws.OPT_RELU, int(layer["relu"]))
    plan.set_option(gdws.OPT_OUT_DTYPE, int(layer["out_f32"]))
    dw, pw = normal((G, s.k, s.k), 1.0 / s.k), normal((s.D, G), 1.0 / math.sqrt(G))
    bias = torch.randn((s.D,), generator=gen, device="cuda") * 0.1
    if not f32 and layer["kind"] != "weights":
        plan.pack_weights(dw, pw, bias)
    x = normal(_shape(s.layout, s.N, s.C, s.H, s.W), 1.0) if with_x else None
    y = torch.empty(_shape(s.layout, s.N, s.D, s.Ho, s.Wo), dtype=torch.float32 if layer["out_f32"] else dtype, device="cuda")
    return {"plan": plan, "x": x, "y": y, "dw": dw, "pw": pw, "bias": bias, "layout": s.layout}


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    layers = _layers(case)
    states = [_prepare_layer(layer, gen, i == 0) for i, layer in enumerate(layers)]
    for prev, st in zip(states, states[1:]):
        st["x"] = prev["y"]
    state = dict(states[0], kind=case["kind"], f32=layers[0]["dtype"] == "f32", layers=states)
    if case["kind"] == "stages":
        s = _spec(case)
        state["z"] = torch.empty((s.N * s.Ho * s.Wo, state["plan"].info()[1]), dtype=torch.bfloat16, device="cuda")
    if case["kind"] == "host":
        state["x"] = state["x"].cpu().pin_memory()
        state["y"] = torch.empty(state["y"].shape, dtype=state["y"].dtype, pin_memory=True)
    return state


def run(state):
    kind, plan = state["kind"], state["plan"]
    if kind == "chain":
        for st in state["layers"]:
            st["plan"].forward(st["x"], st["y"], "NHWC")
        return state["layers"][-1]["y"]
    if kind == "stages":
        plan.depthwise(state["x"], state["z"], "NHWC")
        plan.pointwise(state["z"], state["y"], "NHWC")
        return {"z": state["z"], "y": state["y"]}
    if kind == "host":
        plan.forward_host(state["x"], state["y"], "NHWC")
    elif kind == "weights" or state["f32"]:
        plan.forward(state["x"], state["y"], state["layout"], state["dw"], state["pw"], state["bias"])
    else:
        plan.forward(state["x"], state["y"], state["layout"])
    return state["y"]


def work(case):
    """Each activation and weight once; of the two ways to write the layer (Property 1: k x k filters and a pointwise sum,
    or the k x k convolution they amount to) the one with fewer multiply-adds."""
    size = 4 if case.get("dtype") == "f32" else 2
    total = {"bytes": 0.0, "flops": 0.0}
    for layer in _layers(case):
        s, G = _spec(layer), int(_g(layer).sum())
        px, k2 = s.N * s.Ho * s.Wo, s.k * s.k
        total["bytes"] += size * (s.N * s.H * s.W * s.C + G * (k2 + s.D)) + 4 * s.D
        total["bytes"] += px * s.D * (4 if layer["out_f32"] else size)
        macs = G * (k2 + s.D) if case["kind"] == "stages" else min(G * (k2 + s.D), s.C * k2 * s.D)
        total["flops"] += 2.0 * px * macs
        if case["kind"] == "stages":      # z is written by one call and read by the other
            total["bytes"] += 2 * size * px * G
    return total


def tolerance(case):
    if case.get("dtype") == "f32":
        return {"rel": 1e-5}              # sums of some thousand fp32 products
    # bf16: operands and result are rounded to 8 significant bits, sums are fp32; in a chain 16 such layers follow each other
    return {"rel": 2e-2 if case["kind"] == "chain" else 1e-2}
