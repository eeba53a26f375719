"""Performance cases: what a user of the framework has it do, at the sizes that occur in use.

A case is a dict of plain values.  Its "kind" says which part of the path it is:

  linear   a quantized linear layer (W4A8, W8A8, or weight-only W{2,3,4,8}A16), calibrated activation scale
  asym     a linear layer whose asymmetric activation range is taken from the tensor itself, then the layer
  qkv      self-attention's three projections on one tensor: its scale, one quantization pass, three GEMMs on the codes
  kv       the K and V projections of a cross-attention block, BOS-aware
  conv     a 3x3 convolution (W4A8, W8A8, or weight-only), stride 1 or 2, any image size
  split    a layer fed by a concatenation of two branches with an activation scale for each (shortcut-splitting)
  pack     a layer's weights to their packed form: range, scale and zero-point per channel, codes, layout
  step     one pass over every quantized layer of the SDXL-turbo-shaped UNet

prepare() makes the inputs and what a program keeps beside them (packed weights, scales, a workspace); run() is one pass.
"""
from __future__ import annotations

import math

import torch

from paper_2405_17873_b200 import mixdq, synth
from paper_2405_17873_b200.unet_sweep import UNetSweep

TEXT_DIM = synth.TEXT_DIM
TOKENS = synth.TOKENS_PER_PROMPT


def listed():
    return [
        # one small W8A8 layer: the configuration that the tests and the benchmark start from; launches and latency
        dict(name="linear-256x320x320-w8a8", kind="linear", M=256, N=320, K=320, w_bits=8, act_bits=8),
        # the most frequent layer of the UNet: attention projection of the 1280-channel level, four images
        dict(name="attn-1024x1280x1280-w4a8", kind="linear", M=1024, N=1280, K=1280, w_bits=4, act_bits=8),
        # dynamic asymmetric activations (the paper's quantizer) on the 640-channel level, four images
        dict(name="asym-4096x640x640-w8a8", kind="asym", M=4096, N=640, K=640, w_bits=8),
        # dynamic per-tensor scale shared by q, k and v
        dict(name="qkv-1024x1280x1280-w4a8", kind="qkv", M=1024, N=1280, K=1280, w_bits=4),
        # text conditioning of one cross-attention block for eight prompts
        dict(name="kv-8x1280-w4a8", kind="kv", B=8, N=1280, w_bits=4),
        # the largest convolution of the 512-pixel UNet, four images
        dict(name="conv-4x64x64-640-640-w4a8", kind="conv", B=4, H=64, W=64, Cin=640, Cout=640, stride=1, w_bits=4, act_bits=8),
        # the same level of a picture that is not 512 pixels square (768: 96, 48 and 24 pixels a side)
        dict(name="conv-1x48x48-640-640-w8a8", kind="conv", B=1, H=48, W=48, Cin=640, Cout=640, stride=1, w_bits=8, act_bits=8),
        # a residual convolution of the up path on [hidden | skip]
        dict(name="split-4x16x16-2560-1280-w4a8", kind="split", B=4, H=16, W=16, Cin=2560, split_at=1280, Cout=1280, taps=9, w_bits=4),
        # weight-only on few rows: the weights' bytes are the work
        dict(name="ffn-16x10240x1280-w4a16", kind="linear", M=16, N=10240, K=1280, w_bits=4, act_bits=16),
        # weight-only on an image's rows
        dict(name="attn-1024x1280x1280-w3a16", kind="linear", M=1024, N=1280, K=1280, w_bits=3, act_bits=16),
        # preparing a checkpoint: the largest linear layer to three bits
        dict(name="pack-10240x1280-w3", kind="pack", N=10240, K=1280, bits=3),
        # the whole UNet's layers, four images, W4A8 with a tenth of the layers at W8A8
        dict(name="step-b4-w4a8", kind="step", B=4, table="w4a8"),
    ]


def _log_int(rng, lo, hi, multiple=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(multiple, int(round(v / multiple)) * multiple)


def _channels(rng, lo, hi, multiple):
    """A channel count: half the time one of the UNet's own, else any multiple inside the range."""
    own = [c for c in (320, 640, 960, 1280, 1920, 2560) if lo <= c <= hi]
    return rng.choice(own) if rng.random() < 0.5 else _log_int(rng, lo, hi, multiple)


def _image(rng, pixels_most):
    """Image batch and size: a power-of-two square half the time, else any height and width from 8 to 96."""
    B = rng.randint(1, 8)
    H = W = rng.choice((16, 32, 64))
    if rng.random() < 0.5:
        H, W = _log_int(rng, 8, 96), _log_int(rng, 8, 96)
    while B > 1 and B * H * W > pixels_most:
        B -= 1
    return B, H, W


def draw(rng):
    kind = rng.choice(("linear", "linear", "linear", "asym", "qkv", "kv", "conv", "conv", "split", "pack", "step"))
    if kind in ("linear", "asym", "qkv"):
        case = dict(kind=kind, M=_log_int(rng, 1, 16384), K=_channels(rng, 320, 5120, 16), w_bits=rng.choice((4, 8)))
        case["N"] = case["K"] if kind == "qkv" else _channels(rng, 320, 10240, 4)
        if kind == "linear":
            case["act_bits"] = rng.choice((8, 16))
            if case["act_bits"] == 16:
                case["w_bits"] = rng.choice((2, 3, 4, 8))
        return case
    if kind == "kv":
        return dict(kind=kind, B=rng.randint(1, 16), N=_channels(rng, 320, 2560, 8), w_bits=rng.choice((4, 8)))
    if kind == "conv":
        Cin, Cout = _channels(rng, 320, 2560, 32), _channels(rng, 320, 1280, 8)
        B, H, W = _image(rng, min(16384, 8_000_000_000 // (Cin * Cout)))  # wide layers run on the smaller images
        end = rng.random()
        if end < 0.1:
            Cin, Cout = 4, 320  # the first layer: latents in
        elif end < 0.2:
            Cin, Cout = 320, 4  # the last one: latents out
        act_bits = rng.choice((8, 8, 16))
        w_bits = 8 if end < 0.2 else rng.choice((4, 8) if act_bits == 8 else (2, 3, 4, 8))
        return dict(kind=kind, B=B, H=H, W=W, Cin=Cin, Cout=Cout, stride=rng.choice((1, 1, 1, 2)) if end >= 0.2 else 1,
                    w_bits=w_bits, act_bits=act_bits)
    if kind == "split":
        # the levels of the up path: the call takes images that tile into 128-pixel boxes
        side, Cin, lo, Cout = rng.choice(((16, 2560, 1280, 1280), (16, 1920, 1280, 1280), (32, 1920, 1280, 640), (32, 1280, 640, 640),
                                          (32, 960, 640, 640), (64, 960, 640, 320), (64, 640, 320, 320)))
        return dict(kind=kind, B=rng.randint(1, 8), H=side, W=side, Cin=Cin, split_at=lo, Cout=Cout, taps=rng.choice((1, 9)),
                    w_bits=rng.choice((4, 8)))
    if kind == "pack":
        return dict(kind=kind, N=_channels(rng, 320, 10240, 1), K=_log_int(rng, 320, 11520, 8), bits=rng.choice((2, 3, 4, 8)))
    return dict(kind=kind, B=rng.randint(1, 3), table=rng.choice(("w4a8", "a16")))


# ------------------------------------------------------------------------------------------------ inputs

def _normal(g, *shape, std=1.0):
    return (torch.randn(shape, generator=g, device="cuda") * std).to(torch.float16)


def _activations(g, rows, K):
    """N(0, 1) with one channel in a hundred twenty times as large, as before a transformer's linear layers."""
    x = torch.randn((rows, K), generator=g, device="cuda")
    x[:, torch.randperm(K, generator=g, device="cuda")[: max(1, K // 100)]] *= 20.0
    return x.to(torch.float16)


def _weights(g, N, K, bits, symmetric):
    W = _normal(g, N, K, std=0.02)
    scale, zero = mixdq.weight_minmax_params(W, bits, symmetric)
    zero = None if symmetric else zero
    return W, mixdq.pack_weights(W, bits, scale, zero), scale, zero


def _layer(g, s, N, K, bits, symmetric=True):
    _, s["packed"], s["scale"], s["zero"] = _weights(g, N, K, bits, symmetric)
    s["bias"] = _normal(g, N, std=0.01)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = dict(case=case, status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    return _PREPARE[case["kind"]](case, seed, g, s)


def _prepare_linear(c, seed, g, s):
    s["x"] = _activations(g, c["M"], c["K"])
    _layer(g, s, c["N"], c["K"], c["w_bits"], symmetric=c["act_bits"] == 8)
    s["sx"] = mixdq.act_scale(s["x"]) if c["act_bits"] == 8 else None
    s["ws"] = mixdq.new_workspace(mixdq.workspace_bytes(c["M"], c["N"], c["K"], c["w_bits"], c["act_bits"]))
    return s


def _prepare_asym(c, seed, g, s):
    s["x"] = torch.nn.functional.gelu(_activations(g, c["M"], c["K"]))
    _layer(g, s, c["N"], c["K"], c["w_bits"])
    s["sums"] = mixdq.weight_code_sums(s["packed"], c["N"], c["K"], c["w_bits"])
    s["ws"] = mixdq.new_workspace(mixdq.workspace_bytes(c["M"], c["N"], c["K"], c["w_bits"], 8))
    return s


def _prepare_qkv(c, seed, g, s):
    s["x"] = _activations(g, c["M"], c["K"])
    s["layers"] = []
    for _ in range(3):
        layer = {}
        _layer(g, layer, c["N"], c["K"], c["w_bits"])
        s["layers"].append(layer)
    return s


def _prepare_kv(c, seed, g, s):
    text = _normal(g, c["B"], TOKENS, TEXT_DIM)
    bos = torch.randn(TEXT_DIM, generator=g, device="cuda")
    far = torch.randperm(TEXT_DIM, generator=g, device="cuda")[:8]
    bos[far] = torch.where(bos[far] < 0, -50.0, 50.0)
    text[:, 0, :] = bos.to(torch.float16)
    s["text"] = text
    s["sx"] = mixdq.act_scale(text.reshape(-1, TEXT_DIM), TOKENS)
    s["layers"] = []
    for _ in range(2):
        W, packed, scale, _zero = _weights(g, c["N"], TEXT_DIM, c["w_bits"], True)
        s["layers"].append(dict(packed=packed, scale=scale, bos=synth.bos_projection(text[0, 0], W)))
    s["ws"] = mixdq.new_workspace(mixdq.workspace_bytes(c["B"] * (TOKENS - 1), c["N"], TEXT_DIM, c["w_bits"], 8))
    return s


def _prepare_conv(c, seed, g, s):
    s["x"] = _normal(g, c["B"], c["H"], c["W"], c["Cin"])
    _layer(g, s, c["Cout"], 9 * c["Cin"], c["w_bits"], symmetric=c["act_bits"] == 8)
    s["sx"] = mixdq.act_scale(s["x"]) if c["act_bits"] == 8 else None
    s["ws"] = mixdq.new_workspace(mixdq.conv3x3_workspace_bytes(c["B"], c["H"], c["W"], c["Cin"], c["Cout"], c["stride"],
                                                               c["w_bits"], c["act_bits"]))
    return s


def _prepare_split(c, seed, g, s):
    at, pixels = c["split_at"], c["B"] * c["H"] * c["W"]
    x = _normal(g, c["B"], c["H"], c["W"], c["Cin"])
    x[..., at:] *= 0.25  # the skip connection's range is another one
    s["x"] = x if c["taps"] == 9 else x.reshape(-1, c["Cin"])
    s["s_lo"], s["s_hi"] = mixdq.act_scale(x[..., :at].contiguous()), mixdq.act_scale(x[..., at:].contiguous())
    W = _normal(g, c["Cout"], c["taps"], c["Cin"], std=0.02)
    s["scale"], _ = mixdq.weight_minmax_params(W.reshape(c["Cout"], -1), c["w_bits"], True)
    s["lo"], s["hi"] = (mixdq.pack_weights(part.reshape(c["Cout"], -1).contiguous(), c["w_bits"], s["scale"])
                        for part in (W[:, :, :at], W[:, :, at:]))
    s["bias"] = _normal(g, c["Cout"], std=0.01)
    s["ws"] = mixdq.new_workspace(mixdq.split_workspace_bytes(pixels, c["Cin"], at, pixels, c["Cout"]))
    return s


def _prepare_pack(c, seed, g, s):
    s["w"] = _normal(g, c["N"], c["K"], std=0.02)
    return s


def _step_specs(c):
    specs = synth.unet_layers()
    (synth.assign_bits_w4a8 if c["table"] == "w4a8" else synth.assign_bits_weight_only)(specs)
    return specs


def _prepare_step(c, seed, g, s):
    s["sweep"] = UNetSweep(c["B"], c["table"], seed=seed % 1000003, layers=_step_specs(c))
    return s


_PREPARE = dict(linear=_prepare_linear, asym=_prepare_asym, qkv=_prepare_qkv, kv=_prepare_kv, conv=_prepare_conv,
                split=_prepare_split, pack=_prepare_pack, step=_prepare_step)


# ------------------------------------------------------------------------------------------------ one pass

def run(s):
    return _RUN[s["case"]["kind"]](s["case"], s)


def _run_linear(c, s):
    return mixdq.linear(s["x"], s["packed"], c["N"], c["w_bits"], s["scale"], s["zero"], c["act_bits"], s["sx"], s["bias"],
                        s["ws"], s["status"])


def _run_asym(c, s):
    sx, zx = mixdq.act_asym_params(s["x"])
    y = mixdq.linear_a8_asym(s["x"], s["packed"], c["N"], c["w_bits"], s["scale"], s["sums"], sx, zx, s["bias"], s["ws"],
                             s["status"])
    return dict(scale=sx, zero=zx, y=y)


def _run_qkv(c, s):
    sx = mixdq.act_scale(s["x"])
    codes = mixdq.quantize_acts(s["x"], sx)
    out = [mixdq.linear_q8(codes, l["packed"], c["N"], c["w_bits"], l["scale"], sx, l["bias"], s["status"]) for l in s["layers"]]
    return dict(scale=sx, codes=codes, out=out)


def _run_kv(c, s):
    return [mixdq.crossattn_kv(s["text"], l["packed"], c["N"], c["w_bits"], l["scale"], s["sx"], l["bos"], s["ws"], s["status"])
            for l in s["layers"]]


def _run_conv(c, s):
    return mixdq.conv3x3(s["x"], s["packed"], c["Cout"], c["w_bits"], s["scale"], s["zero"], c["act_bits"], s["sx"], s["bias"],
                         c["stride"], s["ws"], s["status"])


def _run_split(c, s):
    if c["taps"] == 9:
        return mixdq.conv3x3_a8_split(s["x"], c["split_at"], s["lo"], s["hi"], c["Cout"], c["w_bits"], s["scale"], s["s_lo"],
                                      s["s_hi"], s["bias"], 1, s["ws"], s["status"])
    return mixdq.linear_a8_split(s["x"], c["split_at"], s["lo"], s["hi"], c["Cout"], c["w_bits"], s["scale"], s["s_lo"],
                                 s["s_hi"], s["bias"], s["ws"], s["status"])


def _run_pack(c, s):
    symmetric = c["bits"] == 8
    scale, zero = mixdq.weight_minmax_params(s["w"], c["bits"], symmetric)
    return dict(scale=scale, zero=zero, packed=mixdq.pack_weights(s["w"], c["bits"], scale, None if symmetric else zero))


def _run_step(c, s):
    s["sweep"].step()
    return list(s["sweep"].y.values())


_RUN = dict(linear=_run_linear, asym=_run_asym, qkv=_run_qkv, kv=_run_kv, conv=_run_conv, split=_run_split, pack=_run_pack,
            step=_run_step)


# ------------------------------------------------------------------------------------------------ accounting

def _gemm(M, N, K, bits, in_bytes, act_bits=8):
    """Input once, packed weights once, a scale (weight-only: a zero-point too) and a bias per channel, fp16 output once."""
    return dict(bytes=in_bytes + N * K * bits / 8 + N * (6 if act_bits == 8 else 10) + 2 * M * N, flops=2 * M * N * K)


def work(case):
    c, kind = case, case["kind"]
    if kind in ("linear", "asym"):
        return _gemm(c["M"], c["N"], c["K"], c["w_bits"], 2 * c["M"] * c["K"], c.get("act_bits", 8))
    if kind == "qkv":
        one = _gemm(c["M"], c["N"], c["K"], c["w_bits"], 0)
        return dict(bytes=3 * c["M"] * c["K"] + 3 * one["bytes"], flops=3 * one["flops"])
    if kind == "kv":
        one = _gemm(c["B"] * TOKENS, c["N"], TEXT_DIM, c["w_bits"], 0)
        return dict(bytes=2 * c["B"] * TOKENS * TEXT_DIM + 2 * one["bytes"], flops=2 * one["flops"])
    if kind == "conv":
        rows = c["B"] * -(-c["H"] // c["stride"]) * -(-c["W"] // c["stride"])
        return _gemm(rows, c["Cout"], 9 * c["Cin"], c["w_bits"], 2 * c["B"] * c["H"] * c["W"] * c["Cin"], c["act_bits"])
    if kind == "split":
        pixels = c["B"] * c["H"] * c["W"]
        return _gemm(pixels, c["Cout"], c["taps"] * c["Cin"], c["w_bits"], 2 * pixels * c["Cin"])
    if kind == "pack":
        return dict(bytes=c["N"] * (2 * c["K"] + c["K"] * c["bits"] / 8 + 8), flops=4 * c["N"] * c["K"])
    total = dict(bytes=0.0, flops=0.0)
    for l in _step_specs(c):
        in_rows = c["B"] * l.H * l.H if l.H else l.rows(c["B"])
        one = _gemm(l.rows(c["B"]), l.N, l.K, l.w_bits, 2 * in_rows * (l.Cin or l.K), l.a_bits)
        total = {k: total[k] + one[k] for k in total}
    return total


def tolerance(case):
    if case["kind"] == "pack":
        return "exact"
    # integer (or fp32) sums, one fp32 scale and bias step, rounded to fp16: neighbouring fp16 values at most
    return {"rel": 1e-3, "max": 4e-3}
