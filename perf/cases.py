"""The convolution work the performance of this repository is judged by.

``listed()`` holds the twelve cases, ``draw(rng)`` more of the same ranges.  A case is one of

* ``layer``  one square convolution through ``ConvLayerRunner`` (``mnn_conv_plan_ex`` / ``mnn_conv_run``);
* ``rect``   one 1 x k or k x 1 convolution (``mnn_conv_plan_rect`` / ``mnn_conv_run``);
* ``layers`` every convolution of a ResNet-18 forward, layer after layer, each on its own activations, the way a
  program with its own graph (residual additions, branches) calls the library;
* ``net``    the MobileNet-v1 chain through one ``mnn_net_run``.

Plans use the library's frozen cost constants.  Weights are laid out once in ``prepare``, as an inference program
does; inputs are ReLU(N(0,1)) (or N(0,1) where the repository's own configuration says so), weights Kaiming-normal.
"""
from __future__ import annotations

import math

import torch

from paper_2002_12418_b200 import binding as B
from paper_2002_12418_b200 import workloads as W

PRECISION = {"tf32": B.PREC_TF32, "bf16": B.PREC_BF16}
# Bound of a drawn case: half of the multiply-adds (as work() counts them) of the largest listed one, 512 channels at
# 56 x 56 and batch 64.
MAX_DRAWN_FLOPS = 64 * 512 * 512 * 56 * 56 * 9 * 64 // 324


def _layer(name, N, Cin, Cout, H, W_, k, stride=1, pad=0, dilation=1, groups=1, relu=True, bias=True, precision="tf32",
           x="relu_normal"):
    return dict(name=name, kind="layer", N=N, Cin=Cin, Cout=Cout, H=H, W=W_, k=k, stride=stride, pad=pad,
                dilation=dilation, groups=groups, relu=relu, bias=bias, precision=precision, x=x)


def listed():
    return [
        # the smallest call: one 28 x 28 image, 32 channels; latency and launches are all of it
        _layer("conv3x3_32_28_b1", 1, 32, 32, 28, 28, 3, pad=1, relu=False, bias=False, x="uniform"),
        # one image through a network's convolutions, called layer by layer: interactive inference
        dict(name="resnet18_b1", kind="layers", N=1, H=224),
        # one image through a depthwise-separable network planned as a whole: interactive inference
        dict(name="mobilenet_v1_b1", kind="net", N=1, H=224),
        # the same two networks at serving batches
        dict(name="resnet18_b32", kind="layers", N=32, H=224),
        dict(name="mobilenet_v1_b64", kind="net", N=64, H=224),
        # wide 3x3 layers at a large batch, both accuracy classes: the Winograd path at its largest
        _layer("conv3x3_256_56_b64_bf16", 64, 256, 256, 56, 56, 3, pad=1, relu=False, bias=False, precision="bf16", x="normal"),
        _layer("conv3x3_512_56_b64", 64, 512, 512, 56, 56, 3, pad=1, relu=False, bias=False, x="normal"),
        # larger kernels
        _layer("conv5x5_128_28_b64", 64, 128, 128, 28, 28, 5, pad=2, relu=False, bias=False, x="normal"),
        _layer("conv7x7_128_28_b64", 64, 128, 128, 28, 28, 7, pad=3, relu=False, bias=False, x="normal"),
        # the factorised 1 x 7 layers of Inception-v3
        dict(name="conv1x7_192_17_b32", kind="rect", N=32, Cin=192, Cout=192, H=17, W=17, kh=1, kw=7, pad_h=0, pad_w=3,
             relu=True, bias=True, precision="tf32"),
        # odd everything: channel counts off every tile, unaligned rows, a batch of seven
        _layer("conv3x3_100_72_35x45_b7", 7, 100, 72, 35, 45, 3, pad=1),
        # dilated context layer of a dense-prediction head
        _layer("conv3x3_d2_256_28_b16", 16, 256, 256, 28, 28, 3, pad=2, dilation=2),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_layer(rng):
    kind = rng.choice(["dense", "dense", "dense", "dense", "pointwise", "pointwise", "strided", "strided", "dilated",
                       "depthwise", "stem", "grouped"])
    N = _log_int(rng, 1, 64)
    H = _log_int(rng, 7, 112)
    W_ = H if rng.random() < 0.5 else _log_int(rng, 7, 112)
    Cin, Cout = _log_int(rng, 16, 512), _log_int(rng, 16, 512)
    if rng.random() < 0.5:                                # half of the draws have the usual channel counts
        Cin, Cout = (Cin + 15) // 16 * 16, (Cout + 15) // 16 * 16
    if rng.random() < 0.3:
        Cout = Cin
    k, stride, dilation, groups = 3, 1, 1, 1
    if kind == "dense":
        k = rng.choice([3, 3, 3, 5, 7])
    elif kind == "pointwise":
        k = 1
    elif kind == "strided":
        k, stride = rng.choice([1, 3, 3, 5]), 2
    elif kind == "dilated":
        dilation = rng.choice([2, 3])
    elif kind == "depthwise":
        Cout = groups = Cin
        stride = rng.choice([1, 2])
    elif kind == "stem":
        k, stride, Cin, Cout = rng.choice([3, 3, 7]), 2, 3, rng.choice([16, 24, 32, 64])
        H, W_ = 2 * H, 2 * W_
        N = min(N, 32)
    else:
        groups = rng.choice([2, 4, 8])
        Cin, Cout = groups * _log_int(rng, 4, 16), groups * _log_int(rng, 4, 16)
        N, H, W_ = min(N, 8), min(H, 28), min(W_, 28)     # these run the sliding-window kernel
    return _layer("", N, Cin, Cout, H, W_, k, stride, dilation * (k - 1) // 2, dilation, groups, relu=rng.random() < 0.6,
                  bias=rng.random() < 0.6, precision="bf16" if rng.random() < 0.2 else "tf32")


def draw(rng):
    while True:
        u = rng.random()
        if u < 0.7:
            case = _draw_layer(rng)
        elif u < 0.82:
            k, along_w = rng.choice([3, 5, 7, 7]), rng.random() < 0.5
            C = _log_int(rng, 32, 320)
            case = dict(name="", kind="rect", N=_log_int(rng, 1, 64), Cin=C, Cout=C if rng.random() < 0.5 else _log_int(rng, 32, 320),
                        H=rng.randint(8, 35), W=rng.randint(8, 35), kh=1 if along_w else k, kw=k if along_w else 1,
                        pad_h=0 if along_w else k // 2, pad_w=k // 2 if along_w else 0, relu=rng.random() < 0.6,
                        bias=rng.random() < 0.6, precision="tf32")
        elif u < 0.92:
            case = dict(name="", kind="net", N=_log_int(rng, 1, 64), H=rng.choice([128, 160, 192, 224, rng.randint(97, 223)]))
        else:
            case = dict(name="", kind="layers", N=_log_int(rng, 1, 32), H=rng.choice([128, 160, 192, 224, rng.randint(97, 223)]))
        if work(case)["flops"] <= MAX_DRAWN_FLOPS and work(case)["bytes"] <= 1 << 29:
            del case["name"]
            return case


# ---------------------------------------------------------------------------
# Shapes
# ---------------------------------------------------------------------------
def _resized(layers, H):
    """The network's layers for an H x H image instead of 224 x 224."""
    at = {}                                               # extent in the 224 network -> extent here
    at[224] = H
    for l in layers:
        if l.OH not in at and l.H in at:
            at[l.OH] = (at[l.H] + 2 * l.pad - l.k) // l.stride + 1
        if l.name.endswith("stem_7x7s2"):                 # the 3 x 3 stride-2 pooling between the stem and the first stage
            at[56] = (at[112] + 2 - 3) // 2 + 1
    return [W.ConvLayer(l.name, l.N, l.Cin, l.Cout, at[l.H], at[l.H], l.k, l.stride, l.pad, l.dilation, l.groups, l.relu)
            for l in layers]


def _layers_of(case):
    """The square layers of a case (rectangular cases have none)."""
    if case["kind"] == "layer":
        return [W.ConvLayer("layer", case["N"], case["Cin"], case["Cout"], case["H"], case["W"], case["k"], case["stride"],
                            case["pad"], case["dilation"], case["groups"], case["relu"], x_dist=case["x"],
                            bias_dist="normal0.1" if case["bias"] else "zero")]
    if case["kind"] == "layers":
        return _resized(W.config2(case["N"]), case["H"])
    return _resized(W.config3(case["N"]), case["H"])


def _rect_out(case):
    return case["H"] + 2 * case["pad_h"] - case["kh"] + 1, case["W"] + 2 * case["pad_w"] - case["kw"] + 1


def _direct_flops(case):
    if case["kind"] == "rect":
        OH, OW = _rect_out(case)
        return 2 * case["N"] * case["Cout"] * case["Cin"] * OH * OW * case["kh"] * case["kw"]
    return sum(l.direct_flops for l in _layers_of(case))


def work(case):
    """Bytes: inputs, weights and biases read once, outputs written once (of a chain: its first input and its last
    output).  Flops: the multiply-adds of the sliding window, or for stride-1 undilated dense kernels of the cheapest
    Winograd form F(m, k), m <= 6, without its transforms."""
    def reduced(k, axes):
        return min(((m + k - 1) / (m * k)) ** axes for m in (1, 2, 4, 6))

    if case["kind"] == "rect":
        OH, OW = _rect_out(case)
        elems = (case["N"] * case["Cin"] * case["H"] * case["W"] + case["N"] * case["Cout"] * OH * OW +
                 case["Cin"] * case["Cout"] * case["kh"] * case["kw"] + (case["Cout"] if case["bias"] else 0))
        return {"bytes": 4 * elems, "flops": _direct_flops(case) * reduced(max(case["kh"], case["kw"]), 1)}
    layers = _layers_of(case)
    elems, flops = 0, 0.0
    for i, l in enumerate(layers):
        elems += l.Cout * (l.Cin // l.groups) * l.k * l.k + (l.Cout if l.bias_dist != "zero" else 0)
        if case["kind"] != "net" or i == 0:
            elems += l.N * l.Cin * l.H * l.W
        if case["kind"] != "net" or i == len(layers) - 1:
            elems += l.N * l.Cout * l.OH * l.OW
        dense = l.stride == 1 and l.dilation == 1 and l.groups == 1 and l.k > 1
        flops += l.direct_flops * (reduced(l.k, 2) if dense else 1.0)
    return {"bytes": 4 * elems, "flops": flops}


# ---------------------------------------------------------------------------
# State and pass
# ---------------------------------------------------------------------------
def _activations(gen, shape, dist):
    if dist == "uniform":
        return torch.rand(shape, generator=gen, device="cuda") * 2 - 1
    x = torch.randn(shape, generator=gen, device="cuda")
    return x.clamp_(min=0) if dist == "relu_normal" else x


def _weights(gen, shape):
    fan_in = shape[1] * shape[2] * shape[3]
    return torch.randn(shape, generator=gen, device="cuda") * math.sqrt(2.0 / fan_in)


def _bias(gen, n, wanted):
    return torch.randn(n, generator=gen, device="cuda") * 0.1 if wanted else None


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["kind"] == "rect":
        opts = B.make_opts(relu=case["relu"], precision=PRECISION[case["precision"]])
        plan = B.mnn_conv_plan_rect(case["N"], case["Cin"], case["Cout"], case["H"], case["W"], case["kh"], case["kw"],
                                    case["pad_h"], case["pad_w"], opts)
        r = B.ConvLayerRunner(case["N"], case["Cin"], case["Cout"], case["H"], case["W"], max(case["kh"], case["kw"]), plan=plan)
        x = _activations(gen, (case["N"], case["Cin"], case["H"], case["W"]), "relu_normal")
        w = _weights(gen, (case["Cout"], case["Cin"], case["kh"], case["kw"]))
        r.prepare(w)
        y = torch.empty((case["N"], case["Cout"]) + _rect_out(case), device="cuda")
        return [(r, x, w, _bias(gen, case["Cout"], case["bias"]), y)]
    layers = _layers_of(case)
    ws = [_weights(gen, (l.Cout, l.Cin // l.groups, l.k, l.k)) for l in layers]
    bs = [_bias(gen, l.Cout, l.bias_dist != "zero") for l in layers]
    if case["kind"] == "net":
        net = B.NetRunner(case["N"], case["H"], case["H"], layers)
        net.prepare(ws)
        net.bind(ws, bs)
        x = _activations(gen, (case["N"], 3, case["H"], case["H"]), "relu_normal")
        y = torch.empty((case["N"], layers[-1].Cout, layers[-1].OH, layers[-1].OW), device="cuda")
        return net, x, y, ws, bs
    calls = []
    for l, w, b in zip(layers, ws, bs):
        opts = B.make_opts(groups=l.groups, relu=l.relu, precision=PRECISION[case.get("precision", "tf32")])
        r = B.ConvLayerRunner(l.N, l.Cin, l.Cout, l.H, l.W, l.k, l.stride, l.pad, l.dilation, opts)
        r.prepare(w)
        calls.append((r, _activations(gen, (l.N, l.Cin, l.H, l.W), l.x_dist), w, b,
                      torch.empty((l.N, l.Cout, l.OH, l.OW), device="cuda")))
    return calls


def run(state):
    if isinstance(state, tuple):
        net, x, y = state[:3]
        return net.run(x, y)
    return [r.run(x, w, b, y) for r, x, w, b, y in state]


def tolerance(case):
    """Relative 2-norm deviation between two correct evaluations of the same accuracy class: each stays within the
    class's documented bound of the exact result (1e-3 / 1e-2 per layer); the chain of 27
    layers adds deviations up (3.6e-3 from the 64-bit chain measured, single layers 4e-8 .. 5e-4, BF16 class 3e-3)."""
    if case["kind"] == "net":
        return {"rel": 8e-3}
    return {"rel": 1e-2 if case.get("precision") == "bf16" else 1e-3}
