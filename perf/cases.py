"""The calls that performance work on the quantizer is measured by.

Each case is one call of the library on the layers of a model (or on one layer): fp32 weights in
device memory (one case: in host memory), codes, scales and error sums out.  The layer shapes are
those of `workloads.py` - the single convolution, the ResNet-18 / ResNet-50 / MobileNetV2-shaped
models, the mixed-kernel model, the large convolutions - at their own width or with all channel
counts multiplied by a factor (thin and wide variants, whose channel counts are then odd numbers),
and generic stacks of convolutions and linear layers.  The values are seeded and stand in for
trained weights as those of `workloads.py` do: normal, normal with outliers, heavy-tailed, and with
a spread of magnitudes over the output channels; they are drawn on the device, since a large case
holds a third of a billion of them.

Fields of a case:
  layers   "resnet50", "resnet50@0.6" (width factor), or "64x64x3x3" / "2048x2048x3x3*8,10x64x1x1"
  values   recipe of the weights
  bits     2..8
  mode     stages to run: 7 = E|K|C; 1, 3 and 5 are the ablation variants E, E|K and E|C
  sums     per-kernel and per-channel error sums wanted (the default of `alloc_outputs`)
  pack     codes as packed int4
  dequant  "", "fp32" or "bf16": also the quantized weights code * scale
  clip     0, or the factor of the absmax scale that is handed in as the caller's own scale
  call     "layer": squant_quantize_layer (allocates its outputs), "model": squant_quantize_model,
           "handle": a ModelCall that the program keeps, "host": host buffers, pinned
"""
import math

import torch

import paper_2202_07471_b200 as sq
from paper_2202_07471_b200 import workloads as W

_BASE = {"values": "normal", "bits": 4, "mode": 7, "sums": True, "pack": False, "dequant": "", "clip": 0.0, "call": "handle"}
_NETS = ("resnet18", "resnet50", "mobilenetv2", "mixed_kernels")
_ALIGN = 512   # tensors start where a caching allocator would put them


def _case(layers, name=None, **kw):
    c = dict(_BASE, layers=layers, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one small convolution, the call of a user who quantizes layer by layer (latency)
        _case("64x64x3x3", "conv_64", call="layer"),
        # whole models, the library's main use: 4-bit weights with all outputs
        _case("resnet18", "resnet18", values="normal_laplace"),
        _case("resnet50", "resnet50", values="student_t4"),
        # the same model at 6 bits with the quantized weights as bfloat16, to be put back into the network
        _case("resnet50", "resnet50_6bit_bf16", values="student_t4", bits=6, dequant="bf16", call="model"),
        # depthwise and pointwise layers: tiny kernels, many channels
        _case("mobilenetv2", "mobilenetv2"),
        # factorised, grouped and odd-sized kernels
        _case("mixed_kernels", "mixed_kernels", values="normal_laplace", call="model"),
        # linear layers, codes and scales only (what a deployment keeps), 8 bits, one of odd size
        _case("4096x4096x1x1*2,11008x4096x1x1,4096x11008x1x1,1001x1537x1x1", "linear_8bit", bits=8, sums=False),
        # output channels wider than one thread block's shared memory: linear layers on flattened feature maps
        _case("256x100352x1x1,128x65541x1x1,64x8192x3x3", "wide_channels"),
        # the user's own (tighter) scales: clipping, with the fake-quantized fp32 weights of a training loop
        _case("resnet18", "resnet18_own_scales", values="normal_laplace", clip=0.7, dequant="fp32"),
        # one large convolution in the packed format of a deployment
        _case("2048x2048x3x3", "conv_2048_int4", values="normal_chanscale", pack=True, sums=False),
        # eight large convolutions: the bandwidth-bound end
        _case("2048x2048x3x3*8", "conv_2048_x8", values="normal_chanscale"),
        # a whole model from and to host memory
        _case("resnet50", "resnet50_host", values="student_t4", call="host"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("layer", "net", "net", "net", "linear", "conv", "large", "wide", "host"))
    values = rng.choice(("normal", "normal_laplace", "student_t4", "normal_chanscale"))
    bits = rng.choice((2, 3, 4, 4, 4, 5, 6, 8))
    kw = {"values": values, "bits": bits, "sums": rng.random() < 0.7, "pack": bits <= 4 and rng.random() < 0.25,
          "dequant": rng.choice(("", "", "", "fp32", "bf16")), "call": rng.choice(("handle", "model")),
          "mode": rng.choice((7, 7, 7, 7, 7, 7, 7, 1, 3, 5)), "clip": rng.choice((0.0,) * 6 + (0.5, 0.85))}
    if kw["mode"] == 5:
        kw["clip"] = 0.0   # E|C takes the absmax scales
    if kind == "layer":
        kh, kw_ = rng.choice(((1, 1), (3, 3), (3, 3), (5, 5), (7, 7), (1, 7), (3, 1)))
        n = log(1, 1024)
        m = max(1, min(4096, log(4e3, 1e7) // (n * kh * kw_)))
        return _case("%dx%dx%dx%d" % (m, n, kh, kw_), **dict(kw, pack=False, dequant="", clip=0.0, sums=True, call="layer"))
    if kind in ("net", "host"):
        name = "%s@%.3f" % (rng.choice(_NETS), rng.uniform(0.3, 1.0 if kind == "host" else 1.4))
        return _case(name, **(dict(kw, call="host", clip=0.0, mode=7, dequant="") if kind == "host" else kw))
    if kind == "linear":
        shapes = ["%dx%dx1x1" % (log(256, 8192), log(256, 12288)) for _ in range(rng.randint(1, 3))]
    elif kind == "conv":
        shapes = ["%dx%dx3x3" % (log(64, 1024), log(64, 900)) for _ in range(rng.randint(1, 4))]
    elif kind == "large":
        n = rng.randint(912, 2048)
        shapes = ["%dx%dx3x3*%d" % (log(256, 2048), n if rng.random() < 0.3 else n & ~3, rng.randint(1, 5 if kw["mode"] == 7 and not kw["clip"] else 2))]
    else:
        k = rng.choice((1, 1, 9))
        n = log(50000, 200000) if k == 1 else log(4500, 20000)
        shapes = ["%dx%dx%s" % (log(8, 300), n, "1x1" if k == 1 else "3x3")]
        if k == 9 and kw["mode"] == 5:
            kw["mode"] = 7   # E|C ends at one thread block's channel length
    return _case(",".join(shapes), **kw)


def _shapes(layers):
    name, _, factor = layers.partition("@")
    if name in W.WORKLOADS:
        shapes = W.WORKLOADS[name].shapes
        if factor:   # input and output widths alike; the first layer keeps its three input channels
            f = float(factor)
            shapes = [(max(1, round(m * f)), n if n <= 3 else max(1, round(n * f)), kh, kw) for m, n, kh, kw in shapes]
        return [tuple(s) for s in shapes]
    out = []
    for part in layers.split(","):
        dims, _, count = part.partition("*")
        out += [tuple(int(v) for v in dims.split("x"))] * int(count or 1)
    return out


def _weights(shape, values, gen):
    m, n, kh, kw = shape
    std = math.sqrt(2.0 / (n * kh * kw))
    w = torch.empty(shape, device="cuda").normal_(0.0, std, generator=gen)
    if values == "normal_laplace":      # one value in twenty from a Laplace distribution of three times the deviation
        u = torch.rand(shape, device="cuda", generator=gen) - 0.5
        lap = u.sign() * torch.log1p(-2.0 * u.abs()) * (-3.0 * std)
        w = torch.where(torch.rand(shape, device="cuda", generator=gen) < 0.05, lap, w)
    elif values == "student_t4":        # four degrees of freedom, scaled to the same deviation
        u = torch.rand((2,) + shape, device="cuda", generator=gen).clamp_(min=1e-20)
        w /= torch.sqrt((u[0] * u[1]).log_().mul_(-0.5)) * math.sqrt(2.0)
    elif values == "normal_chanscale":  # magnitudes of the output channels spread log-uniformly over a factor of four
        w *= torch.exp2(torch.rand((m, 1, 1, 1), device="cuda", generator=gen) * 2.0 - 1.0)
    return w


def _carve(shapes, dtype, place):
    """Tensors of these shapes in one buffer (so that a model's outputs are a handful of tensors), each
    starting on an allocator's boundary; the gaps are zero."""
    size = torch.empty((), dtype=dtype).element_size()
    offsets, total = [], 0
    for s in shapes:
        offsets.append(total)
        total += -(-math.prod(s) * size // _ALIGN) * _ALIGN // size
    whole = torch.zeros(total, dtype=dtype, **place)
    return whole, [whole[o:o + math.prod(s)].view(s) for o, s in zip(offsets, shapes)]


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shapes = _shapes(case["layers"])
    ws = [_weights(s, case["values"], gen) for s in shapes]
    if case["call"] == "layer":
        return {"case": case, "w": ws[0]}
    host = case["call"] == "host"
    place = {"pin_memory": True} if host else {"device": "cuda"}
    if host:
        _, pinned = _carve(shapes, torch.float32, place)
        for p, w in zip(pinned, ws):
            p.copy_(w)
        ws = pinned
    out = {}

    def carve(key, want, dims, dtype):
        if not want:
            return [None] * len(shapes)
        out[key], parts = _carve(dims, dtype, place)
        return parts

    codes = carve("codes", True, [(s[0], (s[1] * s[2] * s[3] + 1) // 2) if case["pack"] else s for s in shapes], torch.int8)
    scales = carve("scales", True, [(s[0],) for s in shapes], torch.float32)
    kernel_err = carve("kernel_err", case["sums"], [s[:2] for s in shapes], torch.float32)
    channel_err = carve("channel_err", case["sums"], [(s[0],) for s in shapes], torch.float32)
    dequant = carve("dequant", case["dequant"] == "fp32", shapes, torch.float32)
    dequant_bf16 = carve("dequant_bf16", case["dequant"] == "bf16", shapes, torch.bfloat16)
    own = [None] * len(shapes)
    if case["clip"]:
        qmax = 2 ** (case["bits"] - 1) - 1
        own = [(w.abs().amax(dim=(1, 2, 3)) * (case["clip"] / qmax)).contiguous() for w in ws]
    buffers = [sq.LayerBuffers(w, *rest) for w, *rest in zip(ws, codes, scales, kernel_err, channel_err, dequant, own, dequant_bf16)]
    flags = sq.FLAG_NARROW_RANGE | (sq.FLAG_PACK_INT4 if case["pack"] else 0)
    state = {"case": case, "buffers": buffers, "flags": flags, "out": out}
    if case["call"] == "handle":
        state["handle"] = sq.ModelCall(buffers, bits=case["bits"], mode=case["mode"], flags=flags)
    return state


def run(state):
    case = state["case"]
    if case["call"] == "layer":
        b = sq.squant_quantize_layer(state["w"], bits=case["bits"], mode=case["mode"])
        return {"codes": b.codes, "scales": b.scales, "kernel_err": b.kernel_err, "channel_err": b.channel_err}
    if case["call"] == "handle":
        state["handle"].run()
    elif case["call"] == "model":
        sq.squant_quantize_model(state["buffers"], bits=case["bits"], mode=case["mode"], flags=state["flags"])
    else:
        sq.squant_quantize_model_host(state["buffers"], bits=case["bits"], mode=case["mode"], flags=state["flags"])
    return state["out"]


def work(case):
    total = flops = 0
    for m, n, kh, kw in _shapes(case["layers"]):
        nk = n * kh * kw
        total += 4 * m * nk + m * ((nk + 1) // 2 if case["pack"] else nk) + 4 * m
        total += 4 * m * (n + 1) if case["sums"] else 0
        total += {"": 0, "fp32": 4, "bf16": 2}[case["dequant"]] * m * nk
        total += 4 * m if case["clip"] else 0
        flops += 4 * m * nk   # divide, round, subtract, add up
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Every decision is integer arithmetic on one correctly rounded division: the results are defined to the bit.
    return "exact"
