"""The work that programs built on this library have it do, as timed cases over the library's public entry points.

A case is a dict of plain values; `kind` says which entry point it goes through:

  net      one forward pass of a synthetic network from a batch that is already on the GPU (``api.Net.forward``)
  host     one forward pass from page-locked host memory and back to it (``api.HostPipeline``: submit, then wait)
  layer    one dense or depthwise convolution through the single-layer entry points (``api.run_layer``)
  fold     the weight compile step of one Conv-BN block (``api.f8_fold_quantize_fixed``)
  requant  one 32-bit tensor quantised for two consumers (``api.f8_requantize_dual_fixed``)

All results are integer codes and have to be equal: the tolerance is "exact" everywhere.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2202_05239_b200 import api, synth

RESNET50_B256 = 256 * 4.09e9      # multiply-adds of the largest listed case; a drawn case stays below it


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # throughput serving at the benchmark's headline configuration
        {"name": "resnet50_b256", "kind": "net", "net": "resnet50", "batch": 256, "image": 224},
        # latency serving: one image
        {"name": "resnet50_b1", "kind": "net", "net": "resnet50", "batch": 1, "image": 224},
        # whatever a request queue held when the batch was closed, at a smaller resolution
        {"name": "resnet50_b19_160", "kind": "net", "net": "resnet50", "batch": 19, "image": 160},
        # the paper's smaller residual network at a middle batch
        {"name": "resnet18_b64", "kind": "net", "net": "resnet18", "batch": 64, "image": 224},
        # the same network with the paper's own sibling handling (32-bit shortcuts, private formats), odd batch
        {"name": "resnet18_siblings_b33", "kind": "net", "net": "resnet18_siblings", "batch": 33, "image": 224},
        # depthwise-separable networks: throughput and a middle batch
        {"name": "mobilenetv1_b256", "kind": "net", "net": "mobilenetv1", "batch": 256, "image": 224},
        {"name": "mobilenetv2_b64", "kind": "net", "net": "mobilenetv2", "batch": 64, "image": 224},
        # one camera frame from host memory to logits in host memory
        {"name": "mobilenetv2_host_b1", "kind": "host", "net": "mobilenetv2", "batch": 1, "image": 224},
        # a program that calls single layers itself: a layer of the CNN layer sweep ...
        {"name": "conv3x3_28_128_b32", "kind": "layer", "depthwise": False, "batch": 32, "h": 28, "c": 128, "c_out": 128, "k": 3,
         "stride": 1, "res": False},
        # ... and the smallest call there is (one 16 x 16 x 16 tile), where only the cost of a call counts
        {"name": "conv3x3_16_16_b1", "kind": "layer", "depthwise": False, "batch": 1, "h": 16, "c": 16, "c_out": 16, "k": 3,
         "stride": 1, "res": False},
        # the weight compile step of the largest 3x3 block of the residual networks
        {"name": "fold_512x4608", "kind": "fold", "c_out": 512, "k": 4608},
        # a 56 x 56 x 256 sum of an odd batch with two consumers, an element count no vector width divides
        {"name": "requant_dual_29m", "kind": "requant", "n": 37 * 56 * 56 * 256 + 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: batches 1..256 and images 96..256 of every network (odd ones among them),
    layers from 7 x 7 to 112 x 112 with 16..1024 channels, compile steps and requantisations over three decades."""
    kind = rng.choice(["net", "net", "net", "net", "host", "layer", "layer", "depthwise", "fold", "requant"])
    if kind in ("net", "host"):
        name = rng.choice(sorted(synth.NETS))
        macs = {"resnet50": 4.09e9, "resnet18": 1.82e9, "resnet18_siblings": 1.82e9, "mobilenetv1": 0.57e9, "mobilenetv2": 0.31e9}[name]
        batch, image = _log_int(rng, 1, 256 if kind == "net" else 64), rng.randint(96, 256)
        batch = max(1, min(batch, int(0.9 * RESNET50_B256 / (macs * (image / 224.0) ** 2))))
        return {"kind": kind, "net": name, "batch": batch, "image": image}
    if kind == "layer":
        stride, k, h = rng.choice([1, 1, 2]), rng.choice([1, 3]), _log_int(rng, 7, 56)
        c, c_out = 16 * _log_int(rng, 1, 64), 8 * _log_int(rng, 2, 128)
        batch = max(1, min(_log_int(rng, 1, 64), int(0.1 * RESNET50_B256 / (h * h * c * c_out * k * k))))
        return {"kind": "layer", "depthwise": False, "batch": batch, "h": h, "c": c, "c_out": c_out, "k": k, "stride": stride,
                "res": stride == 1 and rng.random() < 0.4}
    if kind == "depthwise":
        c = 8 * _log_int(rng, 4, 120)
        return {"kind": "layer", "depthwise": True, "batch": _log_int(rng, 1, 64), "h": _log_int(rng, 7, 112), "c": c, "c_out": c, "k": 3,
                "stride": rng.choice([1, 2]), "res": False}
    if kind == "fold":
        return {"kind": "fold", "c_out": _log_int(rng, 16, 2048), "k": _log_int(rng, 9, 4608)}
    return {"kind": "requant", "n": _log_int(rng, 30_000, 60_000_000)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _images(case, seed):
    """Normalised signed images in FL 6, as synth.draw_image defines them, drawn on the GPU."""
    z = torch.randn((case["batch"], case["image"], case["image"], 3), generator=_gen(seed), device="cuda")
    return torch.floor(z * 64.0 + 0.5).clamp_(-127, 127).to(torch.int8)


def _activations(shape, gen):
    """Rectified unit Gaussians in FL 5, as synth.draw_unsigned_activation defines them."""
    z = torch.randn(shape, generator=gen, device="cuda")
    return torch.floor(z.abs_() * 32.0 + 0.5).clamp_(0, 255).to(torch.uint8)


def _layer(case, seed):
    rng = np.random.default_rng(seed)
    h, c, c_out, k, dw = case["h"], case["c"], case["c_out"], case["k"], case["depthwise"]
    shape = (c, k, k) if dw else (c_out, k, k, c)
    weight, fl_w = synth.draw_weight(rng, shape, math.sqrt(2.0 / (k * k * (1 if dw else c))))
    bias = synth.draw_bias(rng, c_out, 5 + fl_w)
    return synth.Layer(synth.DWCONV if dw else synth.CONV, "layer", 0, 1 if case["res"] else -1, h, h, c, c_out, k, k, case["stride"],
                       k // 2, synth.U8, synth.U8, synth.U8, 5, fl_w, 5, 5, weight, bias)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "net":
        # a loaded model and one batch of images on the GPU
        return {"kind": kind, "net": api.Net(synth.make_net(case["net"], seed, case["image"]), case["batch"]), "x": _images(case, seed)}
    if kind == "host":
        # a loaded model behind the host pipeline, images and logits in page-locked memory
        layers = synth.make_net(case["net"], seed, case["image"])
        return {"kind": kind, "pipe": api.HostPipeline(layers, case["batch"]), "x": _images(case, seed).cpu().pin_memory(),
                "y": torch.zeros((case["batch"], layers[-1].c_out), dtype=torch.int32).pin_memory()}
    gen = _gen(seed)
    if kind == "layer":
        layer = _layer(case, seed)
        x = _activations((case["batch"], layer.h, layer.w, layer.c), gen)
        res = _activations((case["batch"], layer.ho, layer.wo, layer.c_out), gen) if case["res"] else None
        return {"kind": kind, "layer": layer, "x": x, "res": res, "params": (api.to_device(layer.weight), api.to_device(layer.bias))}
    if kind == "fold":
        c_out, k = case["c_out"], case["k"]
        desc = api.FoldDesc(c_out, k, 5, 0, 24, 0.11, 0.07)
        w = torch.randn((c_out, k), generator=gen, device="cuda") * math.sqrt(2.0 / k)
        vec = [torch.rand(c_out, generator=gen, device="cuda") + 0.5 for _ in range(4)]      # gamma, sigma, beta, mu
        return {"kind": kind, "desc": desc, "w": w, "vec": vec, "w_q": torch.empty((c_out, k), dtype=torch.int8, device="cuda"),
                "bias_q": torch.empty(c_out, dtype=torch.int32, device="cuda"), "fl_w": torch.zeros(1, dtype=torch.int32, device="cuda"),
                "ws": torch.empty(api.f8_fold_workspace_bytes(desc), dtype=torch.uint8, device="cuda")}
    # sums of a layer in format 12: a few hundred codes wide after either quantisation
    n = case["n"]
    acc = (torch.randn(n, generator=gen, device="cuda") * float(1 << 15)).to(torch.int32)
    return {"kind": kind, "acc": acc, "y1": torch.empty(n, dtype=torch.uint8, device="cuda"),
            "y2": torch.empty(n, dtype=torch.int8, device="cuda")}


# ------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "net":
        return state["net"].forward(state["x"])
    if kind == "host":
        state["pipe"].submit(state["x"], state["y"])
        state["pipe"].wait()
        return state["y"]
    if kind == "layer":
        return api.run_layer(state["layer"], state["x"], state["res"], state["params"])
    if kind == "fold":
        api.f8_fold_quantize_fixed(state["desc"], state["w"], *state["vec"], state["w_q"], state["bias_q"], state["fl_w"], state["ws"])
        return [state["w_q"], state["bias_q"], state["fl_w"]]
    api.f8_requantize_dual_fixed(state["acc"], 12, state["y1"], synth.U8, 4, state["y2"], synth.S8, 5)
    return [state["y1"], state["y2"]]


# ------------------------------------------------------------------ what a pass cannot do without

_NET_WORK = {}


def _net_work(name, image):
    if (name, image) not in _NET_WORK:
        layers = synth.make_net(name, 0, image)
        _NET_WORK[name, image] = (synth.net_macs_per_image(layers), sum(l.param_bytes() for l in layers), 4 * layers[-1].c_out)
    return _NET_WORK[name, image]


def work(case):
    kind = case["kind"]
    if kind in ("net", "host"):
        # images, parameters and logits; the tensors between the layers need not leave the chip
        macs, params, out = _net_work(case["net"], case["image"])
        return {"bytes": case["batch"] * (3 * case["image"] ** 2 + out) + params, "flops": 2 * case["batch"] * macs}
    if kind == "layer":
        h, c, c_out, k = case["h"], case["c"], case["c_out"], case["k"]
        ho = (h + 2 * (k // 2) - k) // case["stride"] + 1
        y = case["batch"] * ho * ho * c_out
        taps = k * k * (1 if case["depthwise"] else c)
        return {"bytes": case["batch"] * h * h * c + y * (2 if case["res"] else 1) + c_out * (taps + 4), "flops": 2 * y * taps}
    if kind == "fold":
        n = case["c_out"] * case["k"]
        # scale, statistics (two multiply-adds) and quantisation (scale, round) of every weight
        return {"bytes": 5 * n + 20 * case["c_out"] + 4, "flops": 8 * n}
    return {"bytes": 6 * case["n"], "flops": 4 * case["n"]}


def tolerance(case):
    return "exact"
