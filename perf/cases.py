"""The work that a training step asks of DropIT, as timed cases.

One pass is what DropIT adds to a layer in one training step: the forward half (min-k compression of the layer input into
a cache) and the backward half (the weight gradient from that cache), through the entry points of the package:

  linear  dropit_compress + dropit_weight_grad        an nn.Linear layer's input and incoming gradient
  conv    dropit_compress + dropit_conv_weight_grad   an nn.Conv2d layer's
  mlp     DropITGeluLinear, forward and backward      the autograd layer itself, whose compression takes its statistics
                                                      from the GELU in front of it (the stock products are part of it)

The buffers that a training program keeps from step to step (scratch and the fp32 gradient) are made in `prepare`; the cache is
made by the call, because it is what the step has to hold.  Sizes: ViT-B/16 and ViTDet-B linears, ResNet-50 convolutions
and the single fp32 Linear, i.e. the layer calls of `dropit_inputs`, with the layer kinds next to them in the same networks.
Activation laws are those of `dropit_inputs`: post-normalisation N(0, 1), GELU of it, ReLU of it (half exact zeros); gradients
N(0, 0.02^2).  Not here: the random strategy (a baseline of ablations), 8-bit codes of the retained values, and fp32
convolutions.
"""
from __future__ import annotations

import math

import torch

import paper_2202_13808_b200 as dropit
from paper_2202_13808_b200.nn import DropITGeluLinear

_DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}


def _linear(name, tokens, features_in, features_out, gamma, law="normal", dtype="bf16", fmt="bitmask"):
    return {"name": name, "op": "linear", "M": tokens, "Ca": features_in, "Cz": features_out, "gamma": gamma, "law": law,
            "dtype": dtype, "fmt": fmt}


def _conv(name, batch, channels_in, height, width, channels_out, filt, stride, pad, gamma):
    return {"name": name, "op": "conv", "B": batch, "Ca": channels_in, "H": height, "W": width, "Cz": channels_out, "R": filt,
            "S": filt, "stride": stride, "pad": pad, "gamma": gamma, "law": "relu", "dtype": "bf16", "fmt": "bitmask"}


def listed():
    return [
        # the classifier of ViT-B/16 at batch 64: one class token per image; the smallest layer call of a step
        _linear("vitb_head_64", 64, 768, 1000, 0.9),
        # one fp32 layer with few tokens: full-precision training, latency-bound
        _linear("linear_f32_256x768", 256, 768, 768, 0.9, dtype="f32"),
        # attention projection at batch 3 (3 x 197 tokens, an odd number) with the paper's own coordinate format
        _linear("vitb_proj_591_coo", 3 * 197, 768, 768, 0.9, fmt="index32"),
        # the two MLP layers of ViT-B/16 at batch 64, the ordinary call: narrow input with wide output, and the other way round
        _linear("vitb_fc1", 64 * 197, 768, 3072, 0.9),
        _linear("vitb_fc2", 64 * 197, 3072, 768, 0.9, law="gelu"),
        # detection at 1024 x 1024 pixels, batch 8: the qkv projection at the mildest drop ratio that is used
        _linear("vitdet_qkv_g0.5", 8 * 4096, 768, 2304, 0.5),
        # ... and the second MLP layer, the largest call: 201 MB of input, more than the L2 cache
        _linear("vitdet_fc2_g0.8", 8 * 4096, 3072, 768, 0.8, law="gelu"),
        # ResNet-50 at batch 64, stage 1: the 1x1 and the 3x3 convolution of a bottleneck on 56 x 56 planes
        _conv("r50_conv1x1", 64, 256, 56, 56, 64, 1, 1, 0, 0.8),
        _conv("r50_conv3x3", 64, 64, 56, 56, 64, 3, 1, 1, 0.8),
        # the 3x3 convolution that halves the plane at the start of stage 2
        _conv("r50_conv3x3_stride2", 64, 128, 56, 56, 128, 3, 2, 1, 0.8),
        # stage 3: planes of 14 x 14 (rows are no multiple of 16 bytes), more channels
        _conv("r50_conv3x3_14", 64, 256, 14, 14, 256, 3, 1, 1, 0.8),
        # the autograd layer: GELU + second MLP layer of ViT-B/16 at batch 16, forward and backward
        {"name": "vitb_gelu_fc2_layer", "op": "mlp", "M": 16 * 197, "Ca": 3072, "Cz": 768, "gamma": 0.9, "law": "normal",
         "dtype": "bf16", "fmt": "bitmask"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_MAX_PRODUCT = 32768 * 3072 * 768      # multiply-adds of the largest listed call


def draw(rng):
    gamma = round(rng.uniform(0.5, 0.95), 2)
    kind = rng.choice(("block", "block", "block", "head", "f32", "conv", "conv", "mlp"))
    if kind == "conv":
        # bottleneck layers: plane sides 7 .. 56 (odd ones too), channels in eights, 1x1 or 3x3, stride 1 or 2
        side = _log_int(rng, 7, 56)
        filt, stride = rng.choice(((1, 1), (3, 1), (3, 1), (3, 2), (1, 2)))
        ca, cz = 8 * _log_int(rng, 4, 64), 8 * _log_int(rng, 4, 64)
        batch = _log_int(rng, 2, 64)
        out = (side - 1) // stride + 1
        while batch > 1 and (batch * ca * side * side > 64 * 256 * 56 * 56 or
                             batch * out * out * ca * cz * filt * filt > 64 * 14 * 14 * 256 * 256 * 9):
            batch = (batch + 1) // 2
        case = _conv("", batch, ca, side, side, cz, filt, stride, filt // 2, gamma)
    elif kind == "head":
        # a classifier: one token per image; 10, 100 or 1000 classes
        case = _linear("", _log_int(rng, 8, 512), 8 * _log_int(rng, 24, 128), rng.choice((10, 100, 1000)), gamma)
    elif kind == "f32":
        case = _linear("", _log_int(rng, 64, 1024), 8 * _log_int(rng, 24, 128), 8 * _log_int(rng, 24, 128), gamma, dtype="f32")
    else:
        hidden = 8 * _log_int(rng, 24, 128)             # 192 .. 1024
        tokens = _log_int(rng, 197, 32768)
        ca, cz, law = rng.choice(((hidden, 3 * hidden, "normal"), (hidden, hidden, "normal"), (hidden, 4 * hidden, "normal"),
                                  (4 * hidden, hidden, "gelu")))
        if kind == "mlp":
            ca, cz, tokens = 4 * hidden, hidden, min(tokens, 64 * 197)
        tokens = min(tokens, _MAX_PRODUCT // (ca * cz))
        case = _linear("", tokens, ca, cz, gamma, law, fmt=rng.choice(("bitmask", "bitmask", "bitmask", "index32")))
        if kind == "mlp":
            case.update(op="mlp", law="normal", fmt="bitmask")
    del case["name"]
    return case


def _out_size(case):
    return ((case["H"] + 2 * case["pad"] - case["R"]) // case["stride"] + 1,
            (case["W"] + 2 * case["pad"] - case["S"]) // case["stride"] + 1)


def prepare(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    dtype = _DTYPE[case["dtype"]]

    def normal(shape, std=1.0):
        return torch.randn(shape, generator=gen, device=dev, dtype=torch.float32).mul_(std)

    if case["op"] == "conv":
        ho, wo = _out_size(case)
        x = normal((case["B"], case["Ca"], case["H"], case["W"]))
        dy = normal((case["B"], case["Cz"], ho, wo), 0.02)
    else:
        x = normal((case["M"], case["Ca"]))
        dy = normal((case["M"], case["Cz"]), 0.02)
    if case["law"] == "gelu":
        x = torch.nn.functional.gelu(x)
    elif case["law"] == "relu":
        x = torch.relu(x)
    state = {"case": case, "x": x.to(dtype), "dy": dy.to(dtype)}
    if case["op"] == "mlp":
        layer = DropITGeluLinear(case["Ca"], case["Cz"], gamma=case["gamma"], fmt=case["fmt"], device=dev, dtype=dtype).train()
        with torch.no_grad():
            layer.weight.copy_(normal((case["Cz"], case["Ca"]), case["Ca"] ** -0.5))
            layer.bias.copy_(normal((case["Cz"],), 0.02))
        state["layer"] = layer
        state["x"].requires_grad_(True)
        return state
    code, fmt = (dropit.BF16, dropit.F32)[case["dtype"] == "f32"], (dropit.FMT_BITMASK, dropit.FMT_INDEX32)[case["fmt"] == "index32"]
    n = x.numel()
    state["ws_compress"] = torch.empty(max(dropit.dropit_cache_sizes(n, case["gamma"], code, fmt)[3], 16), dtype=torch.uint8,
                                       device=dev)
    if case["op"] == "conv":
        shape = (case["B"], case["Ca"], case["H"], case["W"], case["Cz"], case["R"], case["S"], case["stride"], case["pad"])
        ws = dropit.dropit_conv_weight_grad_workspace(*shape, code, fmt, dev)
        state["dw"] = torch.empty((case["Cz"], case["Ca"], case["R"], case["S"]), dtype=torch.float32, device=dev)
    else:
        ws = dropit.dropit_weight_grad_workspace(case["M"], case["Ca"], case["Cz"], code, fmt, dev)
        state["dw"] = torch.empty((case["Cz"], case["Ca"]), dtype=torch.float32, device=dev)
    state["ws_grad"] = torch.empty(max(ws, 16), dtype=torch.uint8, device=dev)
    return state


def run(state):
    case = state["case"]
    if case["op"] == "mlp":
        layer, x = state["layer"], state["x"]
        z = layer(x)
        dx, dw, db = torch.autograd.grad(z, (x, layer.weight, layer.bias), state["dy"])
        return {"z": z.detach(), "dx": dx, "dw": dw, "db": db}
    cache = dropit.dropit_compress(state["x"], case["gamma"], case["fmt"], workspace=state["ws_compress"])
    if case["op"] == "conv":
        dw = dropit.dropit_conv_weight_grad(state["dy"], cache, (case["R"], case["S"]), case["stride"], case["pad"],
                                            out=state["dw"], workspace=state["ws_grad"])
    else:
        dw = dropit.dropit_weight_grad(state["dy"], cache, out=state["dw"], workspace=state["ws_grad"])
    return {"values": cache.values, "meta": cache.meta, "offsets": cache.offsets, "dw": dw}


def work(case):
    """Bytes: the layer input and the gradient read once, the cache and the weight gradient written once.  Flops: the
    dense product of the method (dropped entries are zeros in it)."""
    es = 4 if case["dtype"] == "f32" else 2
    if case["op"] == "conv":
        ho, wo = _out_size(case)
        n = case["B"] * case["Ca"] * case["H"] * case["W"]
        ndy, ndw = case["B"] * case["Cz"] * ho * wo, case["Cz"] * case["Ca"] * case["R"] * case["S"]
        flops = 2 * case["B"] * ho * wo * ndw
    else:
        n, ndy, ndw = case["M"] * case["Ca"], case["M"] * case["Cz"], case["Cz"] * case["Ca"]
        flops = 2 * case["M"] * ndw
    if case["op"] == "mlp":
        # x, dz, W, b in; z, dx, dW, db out (the cache is internal to the layer); three products of the same size
        return {"bytes": 2 * (2 * n + 2 * ndy + 2 * ndw + 2 * case["Cz"]), "flops": 3 * flops}
    k = dropit.dropit_keep_count(n, case["gamma"])
    meta = 4 * k if case["fmt"] == "index32" else 4 * ((n + 31) // 32)
    return {"bytes": es * n + es * ndy + es * k + meta + 4 * ((n + 127) // 128) + 4 * ndw, "flops": flops}


def tolerance(case):
    """The cache is exact (whole words and retained values carried over bit by bit); the gradients are sums whose order is
    the implementation's.  Against the same sums in fp64: fp32 gradients are off by up to 1.1e-7; bf16 ones (exact
    products, fp32 accumulators of the tensor cores) by up to 1.2e-5 at 32768 tokens and gamma 0.5; what the autograd
    layer returns is rounded to bf16 and is off by 1.7e-3.  Four times that, and more for the short fp32 sums, where
    other orders of summation differ by a few units in the last place."""
    if case["op"] == "mlp":
        return {"rel": 7e-3}
    return {"rel": 2e-6 if case["dtype"] == "f32" else 5e-5}
