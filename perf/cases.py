"""Performance cases: what programs built on this library ask of it, from one small layer to a whole ResNet-50 stack.

Five kinds of case, all through the public entry points, eagerly, as a program without graphs of its own calls them:

  layer   activations of a producer outside the library -> ebs_pack_acts -> ebs_conv2d_mixed (-> ebs_dequant)
  gemm    a 1x1 convolution whose input planes a previous layer left on the device (matrix product, classifier)
  net     a network object of `network.py`: CIFAR ResNets layer by layer or in one launch, the ImageNet ResNet-18
  stack   the ResNet-50 bottleneck convolutions chained through their packed outputs, with or without shortcuts
  search  the search-stage forward of one layer: meta weights and activations blended over the candidate bitwidths

Inputs are synthetic: half-normal activations, normal weights and smooth noisy images, all from the seed alone.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import torch

from paper_2003_07577_b200 import binding as ebs
from paper_2003_07577_b200 import network

IN_TYPES = {"f32": (ebs.EBS_F32, torch.float32, 4), "u8": (ebs.EBS_U8_CODES, torch.uint8, 1)}
LAYOUTS = {"nchw": ebs.EBS_NCHW, "nhwc": ebs.EBS_NHWC}


# ---------------------------------------------------------------------------------------------------- the cases
def _layer(n, c_in, c_out, k, stride, h, w, w_bits, a_bits, levels, dtype, layout, out):
    return {"kind": "layer", "n": n, "c_in": c_in, "c_out": c_out, "k": k, "stride": stride, "h": h, "w": w,
            "w_bits": w_bits, "a_bits": a_bits, "levels": levels, "dtype": dtype, "layout": layout, "out": out}


def listed():
    return [
        # one small layer, batch 1: the latency of a call chain (pack, convolution with both integer outputs, dequant)
        dict(_layer(1, 64, 64, 3, 1, 32, 32, 2, 2, 0, "u8", "nhwc", "dequant"), name="layer_single_image"),
        # a layer outside every tile size: odd channels, image and batch, the paper's own weight levels, fp32 result
        dict(_layer(7, 45, 77, 3, 1, 29, 37, 3, 5, 1, "f32", "nhwc", "y"), name="layer_ragged_levels"),
        # the first quantized layer of an ImageNet network behind an fp32 NCHW producer, full training-size batch
        dict(_layer(256, 64, 64, 3, 1, 56, 56, 4, 4, 0, "f32", "nchw", "packed"), name="layer_entry_fp32"),
        # ResNet-20 at the batch of its benchmark configuration, layer by layer: 25 short launches
        {"name": "cifar_resnet20_layers", "kind": "net", "net": "cifar", "blocks": 3, "fused": False, "n": 128, "side": 32,
         "bits_seed": 0},
        # the same network in one launch
        {"name": "cifar_resnet20_fused", "kind": "net", "net": "cifar", "blocks": 3, "fused": True, "n": 128, "side": 32,
         "bits_seed": 0},
        # the deepest CIFAR network on a single image: pure latency
        {"name": "cifar_resnet56_one_image", "kind": "net", "net": "cifar", "blocks": 9, "fused": True, "n": 1, "side": 32,
         "bits_seed": 1},
        # ImageNet ResNet-18, one image: interactive serving
        {"name": "resnet18_one_image", "kind": "net", "net": "resnet18", "blocks": 2, "fused": False, "n": 1, "side": 224,
         "bits_seed": 0},
        # ImageNet ResNet-18, batch serving
        {"name": "resnet18_batch64", "kind": "net", "net": "resnet18", "blocks": 2, "fused": False, "n": 64, "side": 224,
         "bits_seed": 0},
        # the headline configuration: the ResNet-50 convolutions of 256 images chained through packed planes
        {"name": "resnet50_stack_256", "kind": "stack", "n": 256, "side": 56, "shortcuts": False, "bits_seed": 0},
        # the same network with folded batch normalisation and its shortcuts, at a serving batch
        {"name": "resnet50_shortcuts_16", "kind": "stack", "n": 16, "side": 56, "shortcuts": True, "bits_seed": 1},
        # one point of the bit-plane GEMM sweep, integer accumulators out
        {"name": "gemm_4096", "kind": "gemm", "h": 64, "w": 64, "c_in": 4096, "c_out": 4096, "w_bits": 4, "a_bits": 4,
         "out": "acc"},
        # one step of the bitwidth search on a mid-network layer, five candidates
        {"name": "search_layer", "kind": "search", "n": 64, "c_in": 128, "c_out": 128, "k": 3, "side": 28, "cand": 5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Half of all layers have whole 32-channel words (networks), the others any count."""
    c = _log(rng, lo, hi)
    return max(32, 32 * round(c / 32)) if rng.random() < 0.5 and hi >= 32 else c


def draw(rng: random.Random):
    kind = rng.choice(["layer", "layer", "layer", "gemm", "gemm", "net", "net", "net", "stack", "search"])
    if kind == "layer":
        c = _layer(_log(rng, 1, 256), _channels(rng, 3, 512), _channels(rng, 10, 512), rng.choice([1, 3, 3, 3, 5]),
                   rng.choice([1, 1, 2]), _log(rng, 7, 112), _log(rng, 7, 112), rng.randint(1, 8), rng.randint(1, 8),
                   int(rng.random() < 0.2), rng.choice(["f32", "u8"]), rng.choice(["nchw", "nhwc"]),
                   rng.choice(["packed", "y", "dequant"]))
        while c["n"] > 1 and (_macs(c) > 2e11 or c["n"] * c["h"] * c["w"] * max(c["c_in"], c["c_out"]) > 1e8):
            c["n"] = (c["n"] + 1) // 2
        return c
    if kind == "gemm":
        c = {"kind": "gemm", "h": _log(rng, 1, 128), "w": _log(rng, 1, 128), "c_in": _channels(rng, 32, 8192),
             "c_out": _channels(rng, 32, 8192), "w_bits": rng.randint(1, 8), "a_bits": rng.randint(1, 8),
             "out": rng.choice(["acc", "y", "packed"])}
        while _macs(c) > 2e11:
            c["h"] = (c["h"] + 1) // 2
        return c
    if kind == "net":
        if rng.random() < 0.6:
            return {"kind": "net", "net": "cifar", "blocks": rng.choice([3, 5, 9]), "fused": rng.random() < 0.5,
                    "n": _log(rng, 1, 1024), "side": 32, "bits_seed": rng.randrange(1000)}
        return {"kind": "net", "net": "resnet18", "blocks": 2, "fused": False, "n": _log(rng, 1, 64),
                "side": 2 * rng.randint(48, 128), "bits_seed": rng.randrange(1000)}
    if kind == "stack":
        c = {"kind": "stack", "n": _log(rng, 1, 256), "side": rng.randint(28, 64), "shortcuts": rng.random() < 0.5,
             "bits_seed": rng.randrange(1000)}
        while c["n"] * c["side"] ** 2 * (2 if c["shortcuts"] else 1) > 256 * 56 * 56:
            c["n"] = (c["n"] + 1) // 2
        return c
    c = {"kind": "search", "n": _log(rng, 1, 256), "c_in": _channels(rng, 16, 512), "c_out": _channels(rng, 16, 512),
         "k": rng.choice([1, 3, 3, 5]), "side": _log(rng, 7, 56), "cand": rng.randint(1, 8)}
    while c["n"] > 1 and c["n"] * c["side"] ** 2 * c["c_in"] > 5e7:
        c["n"] = (c["n"] + 1) // 2
    return c


# ---------------------------------------------------------------------------------------------------- sizes
def _out(h, k, stride, pad):
    return (h + 2 * pad - k) // stride + 1


def _record(name, role, c_in, c_out, k, stride, pad, h, w_bits=8, a_bits=8):
    """One layer of a network: the fields `network.calibrated_plans` reads."""
    return SimpleNamespace(name=name, role=role, c_in=c_in, c_out=c_out, k=k, stride=stride, pad=pad, h_in=h, w_in=h,
                           w_bits=w_bits, a_bits=a_bits, w_scale=0.05, h_out=_out(h, k, stride, pad))


def _basic_net(case):
    """Layers of a CIFAR ResNet-(6 blocks + 2) or of the ImageNet ResNet-18, with per-layer bitwidths."""
    bits = random.Random(case["bits_seed"])
    cifar = case["net"] == "cifar"
    pick = lambda: bits.randint(1, 4) if cifar else bits.randint(2, 6)  # noqa: E731
    side = case["side"]
    if cifar:
        widths, c_in, h, pool, classes = [16, 32, 64], 16, side, None, 10
        layers = [_record("conv1", "first", 3, 16, 3, 1, 1, side)]
    else:
        widths, c_in, pool, classes = [64, 128, 256, 512], 64, (3, 2, 1), 1000
        layers = [_record("conv1", "first", 3, 64, 7, 2, 3, side)]
        h = _out(layers[0].h_out, 3, 2, 1)
    for s, width in enumerate(widths):
        for b in range(case["blocks"]):
            stride, tag, a_in = (2 if s and not b else 1), f"s{s + 1}b{b + 1}", pick()
            c1 = _record(tag + "c1", "conv", c_in, width, 3, stride, 1, h, pick(), a_in)
            layers += [c1, _record(tag + "c2", "conv", width, width, 3, 1, 1, c1.h_out, pick(), pick())]
            if stride == 2:
                layers.append(_record(tag + "ds", "shortcut", c_in, width, 1, 2, 0, h, pick(), a_in))
            c_in, h = width, c1.h_out
    layers.append(_record("fc", "fc", c_in, classes, 1, 1, 0, 1))
    return layers, pool


def _bottleneck_stack(case):
    """The 52 quantized convolutions of ResNet-50 as blocks (c1, c2, c3, ds or None), stride on the 3x3."""
    bits = random.Random(case["bits_seed"])
    pick = lambda: bits.randint(2, 8)  # noqa: E731
    blocks, c_in, h = [], 64, case["side"]
    for s, (width, count) in enumerate(zip([64, 128, 256, 512], [3, 4, 6, 3])):
        for b in range(count):
            stride, tag, a_in = (2 if s and not b else 1), f"s{s + 1}b{b + 1}", pick()
            c1 = _record(tag + "c1", "conv", c_in, width, 1, 1, 0, h, pick(), a_in)
            c2 = _record(tag + "c2", "conv", width, width, 3, stride, 1, h, pick(), pick())
            c3 = _record(tag + "c3", "conv", width, 4 * width, 1, 1, 0, c2.h_out, pick(), pick())
            ds = _record(tag + "ds", "shortcut", c_in, 4 * width, 1, stride, 0, h, pick(), a_in) if not b else None
            blocks.append((c1, c2, c3, ds))
            c_in, h = 4 * width, c2.h_out
    return blocks


def _macs(case):
    if case["kind"] == "layer":
        k, s, p = case["k"], case["stride"], case["k"] // 2
        return case["n"] * _out(case["h"], k, s, p) * _out(case["w"], k, s, p) * case["c_in"] * case["c_out"] * k * k
    if case["kind"] == "gemm":
        return case["h"] * case["w"] * case["c_in"] * case["c_out"]
    layers = _basic_net(case)[0] if case["kind"] == "net" else [L for b in _bottleneck_stack(case) for L in b if L]
    return case["n"] * sum(L.h_out ** 2 * L.c_in * L.c_out * L.k ** 2 for L in layers)


def work(case):
    """Inputs (weights at their own bitwidth) read once and outputs written once; two operations a multiply-add."""
    kind = case["kind"]
    if kind == "layer":
        k, s, p = case["k"], case["stride"], case["k"] // 2
        pixels = case["n"] * _out(case["h"], k, s, p) * _out(case["w"], k, s, p)
        inputs = case["n"] * case["h"] * case["w"] * case["c_in"] * IN_TYPES[case["dtype"]][2]
        weights = case["c_in"] * case["c_out"] * k * k * case["w_bits"] / 8
        planes = pixels * -(-case["c_out"] // 32) * 4 * case["a_bits"]
        fp32 = pixels * case["c_out"] * 4
        out = {"packed": planes, "y": fp32, "dequant": planes + 2 * fp32}[case["out"]]
        return {"bytes": inputs + weights + out, "flops": 2 * _macs(case)}
    if kind == "gemm":
        m = case["h"] * case["w"]
        planes_in = m * -(-case["c_in"] // 32) * 4 * case["a_bits"]
        weights = case["c_in"] * case["c_out"] * case["w_bits"] / 8
        out = m * -(-case["c_out"] // 32) * 4 * case["a_bits"] if case["out"] == "packed" else m * case["c_out"] * 4
        return {"bytes": planes_in + weights + out, "flops": 2 * _macs(case)}
    if kind == "net":
        layers = _basic_net(case)[0]
        weights = sum(L.c_in * L.c_out * L.k ** 2 * L.w_bits / 8 for L in layers)
        return {"bytes": case["n"] * (3 * case["side"] ** 2 + 4 * layers[-1].c_out) + weights, "flops": 2 * _macs(case)}
    if kind == "stack":
        blocks = _bottleneck_stack(case)
        weights = sum(L.c_in * L.c_out * L.k ** 2 * L.w_bits / 8 for b in blocks for L in b if L)
        ends = [blocks[-1][2]] + ([] if case["shortcuts"] else [b[3] for b in blocks if b[3]])
        out = sum(case["n"] * L.h_out ** 2 * L.c_out for L in ends)
        return {"bytes": case["n"] * case["side"] ** 2 * 64 + weights + out, "flops": 2 * _macs(case)}
    acts = case["n"] * case["side"] ** 2 * case["c_in"]
    weights = case["c_in"] * case["c_out"] * case["k"] ** 2
    return {"bytes": 8 * (acts + weights), "flops": (acts + weights) * 6 * case["cand"]}


def tolerance(case):
    if case["kind"] == "search":
        # the blended weights jump by a level where the quantizer's argument sits on a tie, which the last bits of tanh
        # decide; the largest jump (one bit, one candidate) is two, the rms of the result about a half
        return {"rel": 1e-3, "max": 0.999}
    if case["kind"] == "net" or case.get("out") in ("y", "dequant"):
        return {"rel": 1e-5}               # fp32 values; whole numbers stay exact
    return "exact"


# ---------------------------------------------------------------------------------------------------- inputs
def _rng(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _act_codes(shape, bits, g):
    top = (1 << bits) - 1
    z = torch.randn(shape, generator=g, device="cuda").abs_()
    return z.mul_(top / 3.0).add_(0.5).floor_().clamp_(0, top).to(torch.uint8)


def _weight_codes(shape, bits, g):
    half = 1 << (bits - 1)
    z = torch.randn(shape, generator=g, device="cuda")
    return z.mul_(half / 3.0).add_(0.5).floor_().clamp_(-half, half - 1).to(torch.int8)


def _images(n, side, g):
    """Smooth gradients with noise on them, so that pixel statistics differ between images and channels."""
    ramp = torch.linspace(0, 1, side, device="cuda")
    u = torch.rand((3, n, 1, 1, 3), generator=g, device="cuda")
    img = 0.2 + 0.6 * u[0] + 0.6 * (u[1] - 0.5) * ramp.view(1, 1, side, 1) + 0.6 * (u[2] - 0.5) * ramp.view(1, side, 1, 1)
    img = img + 0.08 * torch.randn((n, side, side, 3), generator=g, device="cuda")
    return (img * 255.0 + 0.5).floor_().clamp_(0, 255).to(torch.uint8).contiguous()


def _planes(n, h, w, c, bits):
    return torch.empty(ebs.ebs_packed_act_bytes(n, h, w, c, bits) // 4, dtype=torch.int32, device="cuda")


def _packed_weights(desc, g):
    codes = _weight_codes((desc.c_out, desc.c_in, desc.kh, desc.kw), desc.w_bits, g)
    out = torch.empty(ebs.ebs_packed_weight_bytes(desc) // 4, dtype=torch.int32, device="cuda")
    ebs.ebs_pack_weights(codes, ebs.EBS_I8_CODES, ebs.EBS_NCHW, desc, out)
    return out


def _sigma(desc):
    """Standard deviation of the real-valued result for the weight and activation codes drawn here."""
    half, top = 1 << (desc.w_bits - 1), (1 << desc.a_bits) - 1
    w = max(0.5, half / 3.0) * (2 if desc.w_levels else 1)
    return math.sqrt(desc.c_in * desc.kh * desc.kw) * w * max(0.5, top / 3.0) * desc.w_scale * desc.a_scale


def _conv_state(case, desc, n, h, w, g, out):
    """Weights, outputs and epilogue of a single convolution."""
    ho, wo = ebs.ebs_conv_out_shape(desc, h, w)
    S = SimpleNamespace(case=case, desc=desc, n=n, h=h, w=w, pixels=n * ho * wo, acc=None, y=None, packed=None, epi=None)
    S.pw = _packed_weights(desc, g)
    sigma = _sigma(desc)
    if out in ("acc", "dequant"):
        S.acc = torch.empty((n, ho, wo, desc.c_out), dtype=torch.int32, device="cuda")
    if out == "y":
        S.y = torch.empty((n, ho, wo, desc.c_out), dtype=torch.float32, device="cuda")
        bias = 0.2 * sigma * torch.randn(desc.c_out, generator=g, device="cuda")
        S.epi = ebs.epilogue(None, bias, None, True)
    if out in ("packed", "dequant"):
        S.packed = _planes(n, ho, wo, desc.c_out, desc.a_bits)
        S.epi = ebs.epilogue(None, None, None, True, desc.a_bits, 2.6 * sigma / ((1 << desc.a_bits) - 1))
    return S


def _prepare_layer(case, g):
    k = case["k"]
    desc = ebs.conv_desc(case["c_in"], case["c_out"], k, k, case["stride"], case["stride"], k // 2, k // 2,
                         case["w_bits"], case["a_bits"], 0.05, 0.05, case["levels"])
    n, h, w = case["n"], case["h"], case["w"]
    S = _conv_state(case, desc, n, h, w, g, case["out"])
    shape = (n, case["c_in"], h, w) if case["layout"] == "nchw" else (n, h, w, case["c_in"])
    if case["dtype"] == "f32":
        top = ((1 << case["a_bits"]) - 1) * 0.05
        S.x = torch.randn(shape, generator=g, device="cuda").mul_(top / 2.5)     # negative and clipped values too
    else:
        S.x = _act_codes(shape, case["a_bits"], g)
    S.px = _planes(n, h, w, case["c_in"], case["a_bits"])
    if case["out"] == "dequant":
        S.y = torch.empty((S.pixels, case["c_out"]), dtype=torch.float32, device="cuda")
    return S


def _prepare_gemm(case, g):
    desc = ebs.conv_desc(case["c_in"], case["c_out"], 1, 1, 1, 1, 0, 0, case["w_bits"], case["a_bits"], 0.05, 0.05)
    S = _conv_state(case, desc, 1, case["h"], case["w"], g, case["out"])
    codes = _act_codes((1, case["h"], case["w"], case["c_in"]), case["a_bits"], g)
    S.px = _planes(1, case["h"], case["w"], case["c_in"], case["a_bits"])
    ebs.ebs_pack_acts(codes, ebs.EBS_U8_CODES, ebs.EBS_NHWC, 1, case["c_in"], case["h"], case["w"], case["a_bits"], 1.0,
                      S.px)
    return S


def _prepare_net(case, g):
    layers, pool = _basic_net(case)
    codes = {L.name: _weight_codes((L.c_out, L.c_in, L.k, L.k), L.w_bits, g) for L in layers}
    plans = network.calibrated_plans(layers, codes, _images(8, case["side"], g), pool=pool)
    net = network.FusedBasicBlockNet(plans) if case["fused"] else network.BasicBlockNet(plans, pool=pool)
    return SimpleNamespace(case=case, net=net, images=_images(case["n"], case["side"], g))


def _prepare_stack(case, g):
    """Per convolution: descriptor, weights, output buffers and epilogue, in call order, as a program keeps them."""
    n, blocks = case["n"], _bottleneck_stack(case)
    S = SimpleNamespace(case=case, n=n, calls=[], ends=[], side=case["side"], bits=blocks[0][0].a_bits)
    S.x = _act_codes((n, case["side"], case["side"], 64), S.bits, g)
    S.px = _planes(n, case["side"], case["side"], 64, S.bits)

    def conv(L, src, a_scale, next_bits, spread, relu=True, **shortcut):
        """spread: the result's standard deviation after folded normalisation, or None where there is none."""
        d = ebs.conv_desc(L.c_in, L.c_out, L.k, L.k, L.stride, L.stride, L.pad, L.pad, L.w_bits, L.a_bits, L.w_scale,
                          a_scale)
        scale = bias = None
        sigma = _sigma(d)
        if spread is not None:
            scale = (spread / sigma) * (0.9 + 0.2 * torch.rand(L.c_out, generator=g, device="cuda"))
            bias = 0.1 * spread * torch.randn(L.c_out, generator=g, device="cuda")
            sigma = spread
        out = _planes(n, L.h_out, L.h_out, L.c_out, next_bits) if next_bits else None
        y = None if next_bits else torch.empty((n, L.h_out, L.h_out, L.c_out), dtype=torch.float32, device="cuda")
        step = (3.0 if shortcut else 2.6 * sigma) / ((1 << next_bits) - 1) if next_bits else 0.0
        epi = ebs.epilogue(scale, bias, shortcut.get("residual"), relu, next_bits, step or 1.0,
                           res_packed=shortcut.get("res_packed"), res_bits=shortcut.get("res_bits", 0),
                           res_scale=shortcut.get("res_scale", 0.0))
        S.calls.append((src, L.h_in, _packed_weights(d, g), d, epi, y, out))
        return y, out, step

    wired = case["shortcuts"]
    x, step = S.px, 0.05
    for i, (c1, c2, c3, ds) in enumerate(blocks):
        after = blocks[i + 1][0].a_bits if i + 1 < len(blocks) else 8
        _, t, ts = conv(c1, x, step, c2.a_bits, 1.0 if wired else None)
        _, u, us = conv(c2, t, ts, c3.a_bits, 1.0 if wired else None)
        if not wired:
            if ds is not None:
                S.ends.append(conv(ds, x, step, 8, None)[1])
            _, x, step = conv(c3, u, us, after, None)
        elif ds is not None:
            y, _, _ = conv(ds, x, step, 0, 0.5, relu=False)
            _, x, step = conv(c3, u, us, after, 0.5, residual=y)
        else:
            _, x, step = conv(c3, u, us, after, 0.5, res_packed=x, res_bits=c1.a_bits, res_scale=step)
    S.ends.append(x)
    return S


def _prepare_search(case, g):
    shape = (case["n"], case["side"], case["side"], case["c_in"])
    S = SimpleNamespace(case=case, bits=list(range(1, case["cand"] + 1)))
    S.w = 0.05 * torch.randn((case["c_out"], case["c_in"], case["k"], case["k"]), generator=g, device="cuda")
    S.x = torch.randn(shape, generator=g, device="cuda")
    S.w_hat, S.x_hat = torch.empty_like(S.w), torch.empty_like(S.x)
    S.scratch = torch.zeros(4, dtype=torch.int32, device="cuda")
    soft = torch.softmax(torch.randn((2, case["cand"]), generator=g, device="cuda"), dim=1)
    S.coeff_w, S.coeff_x = soft.tolist()
    return S


PREPARE = {"layer": _prepare_layer, "gemm": _prepare_gemm, "net": _prepare_net, "stack": _prepare_stack,
           "search": _prepare_search}


def prepare(case, seed):
    return PREPARE[case["kind"]](case, _rng(seed))


# ---------------------------------------------------------------------------------------------------- one pass
def run(S):
    case = S.case
    kind = case["kind"]
    if kind == "net":
        return S.net.forward(S.images)
    if kind == "search":
        ebs.ebs_search_weight_forward(S.w, S.bits, S.coeff_w, S.w_hat, S.scratch)
        ebs.ebs_search_act_forward(S.x, 2.0, S.bits, S.coeff_x, S.x_hat)
        return S.w_hat, S.x_hat
    if kind == "stack":
        ebs.ebs_pack_acts(S.x, ebs.EBS_U8_CODES, ebs.EBS_NHWC, S.n, 64, S.side, S.side, S.bits, 1.0, S.px)
        for src, h, pw, desc, epi, y, out in S.calls:
            ebs.ebs_conv2d_mixed(src, S.n, h, h, pw, desc, epi, None, y, out)
        return S.ends
    if kind == "layer":
        ebs.ebs_pack_acts(S.x, IN_TYPES[case["dtype"]][0], LAYOUTS[case["layout"]], S.n, case["c_in"], S.h, S.w,
                          case["a_bits"], 0.05, S.px)
    dequant = case["out"] == "dequant"
    ebs.ebs_conv2d_mixed(S.px, S.n, S.h, S.w, S.pw, S.desc, S.epi, S.acc, None if dequant else S.y, S.packed)
    if dequant:
        ebs.ebs_dequant(S.acc, S.pixels, case["c_out"], ebs.ebs_combined_scale(0.05, 0.05), None, None, True, S.y)
    return [t for t in (S.acc, S.y, S.packed) if t is not None]
