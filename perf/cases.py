"""Performance cases of the sub-bit binary convolution library: what a user has it do, through the package's
public classes and functions, from one small layer on one image to a whole network on a large batch.

A case names an entry point ("op"), a layer or a network of the workload lists, a batch size, the index width
tau, the activation type and the output type:

    layer    SnnConv.forward: one layer, device buffers, path chosen by the library
    host     SnnConv.forward_host: the same with pinned host buffers, copies included
    static   forward_static: one forward pass from host-side layer data, without device allocation
    group    SnnConvGroup.forward: all layers of a network, each on its own input, one launch
    stack    SnnConvStack.forward: all layers of a network as a dependent chain, one launch

Layers, codebooks, indices, scales and activations follow the distributions of the workload generators: distinct
random codes, uniform indices, scales in [0.5, 1.5), Bernoulli(1/2) signs or standard-normal fp16 activations.
The thresholds between the layers of a chain (a folded batch normalisation) are normal with half the standard
deviation of the sums they shift, so that both signs occur in every channel.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2110_09195_b200 as snn
import workloads as wl

NETS = {"resnet18": wl.resnet18_layers, "resnet34": wl.resnet34_layers, "resnet20": wl.resnet20_layers,
        "resnet50_1x1": wl.resnet50_1x1_layers}
OUT = {"f32": snn.OUT_F32, "i32": snn.OUT_I32, "signs": snn.OUT_BITS}


def _layer_case(name, op, c_in, c_out, h, w, n, tau, act="bin", out="f32", stride=1, pad=1, ksize=3):
    case = {"op": op, "c_in": c_in, "c_out": c_out, "h": h, "w": w, "stride": stride, "pad": pad, "ksize": ksize,
            "n": n, "tau": tau, "act": act, "out": out}
    return {"name": name, **case} if name else case


def _net_case(name, op, net, n, tau, act="bin", out="f32"):
    case = {"op": op, "net": net, "n": n, "tau": tau, "act": act, "out": out}
    return {"name": name, **case} if name else case


def listed():
    return [
        # the smallest call: one CIFAR-sized layer on one image, as an interactive program makes it
        _layer_case("layer_16ch_1img", "layer", 16, 16, 32, 32, 1, 5),
        # one layer of the third ImageNet stage on a batch: the layer the tau sweep is quoted on
        _layer_case("layer_256ch_n64", "layer", 256, 256, 14, 14, 64, 5),
        # odd channel counts and map, stride 2, the pre-scale sums: layers that fit no tile
        _layer_case("layer_ragged_i32", "layer", 70, 90, 45, 37, 9, 6, out="i32", stride=2),
        # the weights-only deployment of one layer at a small batch
        _layer_case("layer_f16_n8", "layer", 128, 128, 28, 28, 8, 4, act="f16"),
        # a program whose data live in host memory: copies in and out are part of the call
        _layer_case("host_64ch_n16", "host", 64, 64, 56, 56, 16, 5),
        # a program that lets no library allocate device memory: the layer's stored form goes in with every call
        _layer_case("static_128ch_n8", "static", 128, 128, 28, 28, 8, 5),
        # all layers of the benchmark's network at the benchmark's batch
        _net_case("group_resnet18_n64", "group", "resnet18", 64, 5),
        # the same network with fp16 activations
        _net_case("group_resnet18_f16_n64", "group", "resnet18", 64, 5, act="f16"),
        # the CIFAR network: many small layers of few channels
        _net_case("group_resnet20_n128", "group", "resnet20", 128, 6),
        # the bottleneck network's 1x1 layers: the most output bytes
        _net_case("group_resnet50_1x1_n64", "group", "resnet50_1x1", 64, 5),
        # whole-network inference, every layer fed by the one before: one image (latency) ...
        _net_case("stack_resnet18_1img", "stack", "resnet18", 1, 5),
        # ... and the deepest network on a large batch (the most arithmetic)
        _net_case("stack_resnet34_n128", "stack", "resnet34", 128, 5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("layer", "layer", "layer", "group", "group", "group", "stack", "stack", "static", "host"))
    tau = rng.randint(1, 9)
    if op == "group":
        net = rng.choice(tuple(NETS))
        act = "f16" if net in ("resnet18", "resnet20") and rng.random() < 0.35 else "bin"
        out = "f32" if act == "f16" else rng.choice(("f32", "f32", "signs", "i32"))
        return _net_case(None, op, net, _log_int(rng, 1, 128 if net == "resnet20" else 64),
                         min(tau, 8) if net == "resnet50_1x1" else tau, act, out)
    if op == "stack":
        return _net_case(None, op, rng.choice(("resnet18", "resnet34", "resnet20")), _log_int(rng, 1, 96), tau)
    ksize = 1 if op == "layer" and rng.random() < 0.25 else 3
    act = "f16" if op != "static" and rng.random() < 0.3 else "bin"
    out = "f32" if act == "f16" else rng.choice(("f32", "f32", "i32") if op == "static" else ("f32", "f32", "i32", "signs"))
    c_in, c_out = _log_int(rng, 16, 512), _log_int(rng, 16, 512)
    if ksize == 1:
        c_in, tau = (c_in + 7) // 8 * 8, min(tau, 8)
    elif rng.random() < 0.5:   # half of the layers have the round channel counts of the networks, the others any
        c_in, c_out = 1 << int(math.log2(c_in)), 1 << int(math.log2(c_out))
    h, w = _log_int(rng, 6, 57), _log_int(rng, 6, 57)
    n = _log_int(rng, 1, 64 if op == "layer" else 16)
    stride = rng.choice((1, 1, 1, 2))
    pad = 0 if ksize == 1 else rng.choice((1, 1, 1, 0))
    case = _layer_case(None, op, c_in, c_out, h, w, n, tau, act, out, stride, pad, ksize)
    # a large layer on a smaller batch: copies over the host link, popcounts and fp16 products cost more per unit
    most = {"host": (16e6, 4e10), "static": (2e8, 3e10)}.get(op, (4e8, 2e11))
    while case["n"] > 1 and (work(case)["bytes"] > most[0] or work(case)["flops"] > most[1]):
        case["n"] //= 2
    return case


def _shapes(case):
    if "net" in case:
        return NETS[case["net"]]()
    return [wl.LayerShape(case["c_in"], case["c_out"], case["h"], case["w"], case["stride"], case["pad"], case["ksize"])]


def _params(shape, tau, rng):
    """The stored form of a layer: codebook, packed uniform indices (uniform bits), scales."""
    space = 512 if shape.ksize == 3 else 256
    codebook = rng.permutation(space)[:1 << tau].astype(np.uint16)
    units = shape.c_out * (shape.c_in if shape.ksize == 3 else shape.c_in // 8)
    idx_packed = rng.integers(0, 256, size=(units * tau + 7) // 8, dtype=np.uint8)
    alpha = rng.uniform(0.5, 1.5, size=shape.c_out).astype(np.float32)
    return codebook, idx_packed, alpha


def _activations(shape, n, act, gen):
    if act == "f16":
        return torch.randn((n, shape.h, shape.w, shape.c_in), dtype=torch.float16, device="cuda", generator=gen)
    words = (shape.c_in + 31) // 32
    bits = torch.randint(-2 ** 31, 2 ** 31, (n, shape.h, shape.w, words), dtype=torch.int32, device="cuda", generator=gen)
    if shape.c_in % 32:
        bits[..., -1] &= (1 << (shape.c_in % 32)) - 1   # the unused high bits are zero
    return bits


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    op, n, tau, act = case["op"], case["n"], case["tau"], case["act"]
    out_type, act_type = OUT[case["out"]], snn.ACT_F16 if act == "f16" else snn.ACT_BIN
    shapes = _shapes(case)
    state = {"op": op, "out_type": out_type}
    if op == "static":
        s = shapes[0]
        x = _activations(s, n, act, gen)
        out = torch.empty((n, s.h_out, s.w_out, s.c_out), dtype=torch.float32 if out_type == snn.OUT_F32 else torch.int32,
                          device="cuda")
        codebook, idx_packed, alpha = _params(s, tau, rng)
        return {**state, "args": (s.c_in, s.c_out, tau, codebook, idx_packed, alpha, x, out, s.stride, s.pad, out_type)}
    layers = []
    for s in shapes:
        codebook, idx_packed, alpha = _params(s, tau, rng)
        shift = None
        if op == "stack" or case["out"] == "signs":
            shift = (0.5 * math.sqrt(s.ksize * s.ksize * s.c_in) * rng.standard_normal(s.c_out)).astype(np.float32)
        layers.append(snn.SnnConv(s.c_in, s.c_out, tau, codebook, idx_packed, alpha, s.stride, s.pad, act_type,
                                  shift=shift, ksize=s.ksize))
    if op == "group":
        g = snn.SnnConvGroup(layers, [(n, s.h, s.w) for s in shapes])
        return {**state, "group": g, "x": [_activations(s, n, act, gen) for s in shapes], "out": g.alloc_outs(out_type)}
    first = shapes[0]
    x = _activations(first, n, act, gen)
    if op == "stack":
        st = snn.SnnConvStack(layers, n, first.h, first.w)
        return {**state, "stack": st, "x": x, "out": st.alloc_out(out_type)}
    layer = layers[0]
    if op == "host":
        return {**state, "layer": layer, "x": x.cpu().pin_memory(),
                "out": layer.alloc_out(n, first.h, first.w, out_type, pin=True)}
    return {**state, "layer": layer, "x": x, "out": layer.alloc_out(n, first.h, first.w, out_type)}


def run(state):
    op, out_type = state["op"], state["out_type"]
    if op == "layer":
        return state["layer"].forward(state["x"], out=state["out"], out_type=out_type)
    if op == "group":
        return state["group"].forward(state["x"], state["out"], out_type=out_type)
    if op == "stack":
        return state["stack"].forward(state["x"], state["out"], out_type=out_type)
    if op == "static":
        return snn.forward_static(*state["args"])
    return state["layer"].forward_host(state["x"], out=state["out"], out_type=out_type)


def work(case):
    """Inputs and stored weights (index stream, codebook, scales) read once, outputs written once; two operations per
    multiply-accumulate of the dense convolution."""
    n, tau = case["n"], case["tau"]
    shapes = _shapes(case)
    total, macs = 0, 0
    for i, s in enumerate(shapes):
        units = s.c_out * (s.c_in if s.ksize == 3 else s.c_in // 8)
        total += (units * tau + 7) // 8 + 2 * (1 << tau) + 4 * s.c_out
        macs += s.dense_macs(n)
        if case["op"] != "stack" or i == 0:
            total += s.in_bytes_f16(n) if case["act"] == "f16" else s.in_bytes_bin(n)
        if case["op"] != "stack" or i == len(shapes) - 1:
            px = n * s.h_out * s.w_out
            total += px * 4 * ((s.c_out + 31) // 32) if case["out"] == "signs" else px * 4 * s.c_out
    return {"bytes": total, "flops": 2 * macs}


def tolerance(case):
    # Binary activations: the sums are integers, and every fp32 output is one rounding of an exact product.
    if case["act"] == "bin":
        return "exact"
    # fp16 activations: products are exact, sums are fp32 in another order.  Against the same convolution in 64 bits
    # the largest layers (512 input channels) measure 4.6e-7 and 2.7e-6; four times that.
    return {"rel": 2e-6, "max": 1.2e-5}
