"""Timed cases of the binarized-convolution library: the calls that a user's program makes, over the sizes it makes them at.

A case is a dict of plain values; `op` says which call it is:

  net    a Bi-Real Net 18 forward of N images, with the 7x7 stem ("conv7") or the STEM module ("module")
  layer  one binary layer as a network runs it: binarize + pack the fp32 activations, then the convolution with its int32
         sums ("int32") or with the fused BN + sign + re-pack ("sign"); "bits" calls the convolution on packed weights,
         "tensor" the one on weights expanded beforehand
  block  a Bi-Real block on packed activations: convolution + BN + residual add + sign, fp32 stream and packed signs out
  pack   binarize + pack alone
  host   one binary layer with host buffers in and out (copies included)

Sizes are those of Bi-Real Net 18 / ResNet-18 (64 to 512 channels at 56 to 7 pixels, batch 1 to 256), of the large-batch and
bit-pack benchmarks, and odd ones around them.
"""
from __future__ import annotations

import math

import torch

from paper_1908_05858_b200 import binding as B

STAGE_C = (64, 128, 256, 512)
STAGE_HW = (56, 28, 14, 7)


# ---- the cases --------------------------------------------------------------------------------------------------------
def _net(N, stem):
    return {"op": "net", "N": N, "stem": stem}


def _layer(N, C, H, W, O, k, stride, pad_value, layout, engine, out):
    return {"op": "layer", "N": N, "C": C, "H": H, "W": W, "O": O, "k": k, "stride": stride, "pad": k // 2,
            "pad_value": pad_value, "layout": layout, "engine": engine, "out": out}


def _block(N, C, HW, O, stride, engine):
    return {"op": "block", "N": N, "C": C, "HW": HW, "O": O, "stride": stride, "engine": engine}


def _pack(N, C, H, W, layout):
    return {"op": "pack", "N": N, "C": C, "H": H, "W": W, "layout": layout}


def _host(N, C, HW, O, k):
    return {"op": "host", "N": N, "C": C, "HW": HW, "O": O, "k": k}


def listed():
    return [
        # classifying one image as it arrives: latency and launches
        dict(_net(1, "conv7"), name="net_b1"),
        # a small serving batch
        dict(_net(8, "conv7"), name="net_b8"),
        # throughput: a data set classified in large batches
        dict(_net(128, "conv7"), name="net_b128"),
        # the same network with the STEM module, a middling batch
        dict(_net(32, "module"), name="net_module_b32"),
        # the smallest layer, one image: what a call costs at all
        dict(_layer(1, 64, 14, 14, 64, 3, 1, -1, "NCHW", "bits", "int32"), name="layer_b1_c64"),
        # the deepest stage of the network at batch 64, feeding another binary layer
        dict(_layer(64, 512, 7, 7, 512, 3, 1, -1, "NCHW", "bits", "sign"), name="layer_b64_c512"),
        # the large-batch 3x3 layer with its raw sums
        dict(_layer(256, 256, 28, 28, 256, 3, 1, -1, "NCHW", "bits", "int32"), name="layer_b256_c256"),
        # the large-batch pointwise layer (wide output) on expanded weights, feeding another binary layer
        dict(_layer(256, 512, 14, 14, 2048, 1, 1, -1, "NCHW", "tensor", "sign"), name="layer_b256_1x1"),
        # sizes that divide nothing: channel tails, odd images, stride 2, channels-last activations
        dict(_layer(37, 100, 27, 29, 70, 3, 2, +1, "NHWC", "bits", "int32"), name="layer_odd_s2"),
        # a first-stage block of the network, for a program that builds its own
        dict(_block(64, 64, 56, 64, 1, "tensor"), name="block_b64_c64"),
        # packing a large activation tensor (memory-bound)
        dict(_pack(128, 256, 56, 56, "NCHW"), name="pack_128x256x56x56"),
        # host buffers in and out: PCIe and overlap
        dict(_host(64, 256, 28, 256, 3), name="host_b64_c256"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _out(H, k, stride, pad):
    return (H + 2 * pad - k) // stride + 1


def draw(rng):
    while True:
        op = rng.choice(["net"] * 4 + ["layer"] * 5 + ["block", "pack", "host"])
        if op == "net":
            c = _net(_log(rng, 1, 128), rng.choice(["conv7", "conv7", "conv7", "module"]))
            if c["stem"] == "module":
                c["N"] = min(c["N"], 112)
            return c
        if op == "layer":
            C = rng.choice([rng.choice(STAGE_C), _log(rng, 16, 512)])
            O = rng.choice([C, rng.choice(STAGE_C), _log(rng, 16, 2048)])
            H = rng.choice([rng.choice(STAGE_HW), rng.randint(5, 57)])
            W = rng.choice([H, H, max(5, H + rng.randint(-3, 3))])
            k, stride = rng.choice([3, 3, 1]), rng.choice([1, 1, 2])
            c = _layer(_log(rng, 1, 256), C, H, W, O, k, stride, rng.choice([-1, -1, 1]), rng.choice(["NCHW", "NCHW", "NHWC"]),
                       rng.choice(["bits", "bits", "tensor"]), rng.choice(["int32", "sign"]))
        elif op == "block":
            s = rng.randrange(4)
            stride = 2 if s < 3 and rng.random() < 0.25 else 1
            c = _block(_log(rng, 1, 128), STAGE_C[s], STAGE_HW[s] + rng.choice([0, 0, -1, 1]), STAGE_C[s] * stride, stride,
                       rng.choice(["bits", "tensor", "tensor"]))
        elif op == "pack":
            H = rng.choice([rng.choice(STAGE_HW), rng.randint(5, 57)])
            c = _pack(_log(rng, 1, 256), rng.choice([rng.choice(STAGE_C), _log(rng, 16, 512)]), H, rng.choice([H, H + rng.randint(0, 3)]),
                      rng.choice(["NCHW", "NCHW", "NHWC"]))
        else:
            s = rng.randrange(4)
            c = _host(_log(rng, 1, 64), STAGE_C[s], STAGE_HW[s], rng.choice([STAGE_C[s], _log(rng, 16, 512)]), rng.choice([3, 3, 1]))
        w = work(c)
        if w["flops"] <= 1.2e11 * 2 and w["bytes"] <= 4.3e8 and (op != "host" or w["bytes"] <= 1.1e8):
            return c


# ---- what a program has in hand before the call ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _bn(g, O):
    """gamma ~ U(0.5, 1.5), beta ~ N(0, 0.1), running mean ~ N(0, 0.1), running var ~ U(0.5, 1.5)."""
    u = lambda: torch.rand(O, device="cuda", generator=g) + 0.5  # noqa: E731
    n = lambda: 0.1 * torch.randn(O, device="cuda", generator=g)  # noqa: E731
    return u(), n(), n(), u()


def _activations(g, N, C, H, W, layout):
    x = torch.randn((N, C, H, W) if layout == "NCHW" else (N, H, W, C), device="cuda", generator=g)
    x[torch.rand(x.shape, device="cuda", generator=g) < 0.01] = 0.0  # activations hold some exact zeros
    return x


def _weights(g, O, C, k):
    return torch.randn((O, C, k, k), device="cuda", generator=g)


def _net_params(g, module):
    def fp32(*shape):
        fan_in = math.prod(shape[1:])
        return torch.randn(shape, device="cuda", generator=g) / math.sqrt(fan_in)

    p = {"bn_eps": 1e-5, "stem_w": fp32(64, 3, 7, 7), "stem_bn": _bn(g, 64), "block_w": [], "block_bn": [], "down_w": [], "down_bn": []}
    C = 64
    for b in range(16):
        O = STAGE_C[b // 4]
        p["block_w"].append(_weights(g, O, C, 3))
        p["block_bn"].append(_bn(g, O))
        if b % 4 == 0 and b > 0:
            p["down_w"].append(fp32(O, C))
            p["down_bn"].append(_bn(g, O))
        C = O
    p["fc_w"], p["fc_b"] = fp32(1000, 512), 0.1 * torch.randn(1000, device="cuda", generator=g)
    if module:
        shapes = ((32, 3, 3, 3), (16, 32, 1, 1), (32, 16, 3, 3), (64, 64, 1, 1))
        p["stem_module"] = {"w": [fp32(*s) for s in shapes], "bn": [_bn(g, s[0]) for s in shapes]}
    return p


def prepare(case, seed):
    g = _gen(seed)
    op = case["op"]
    s = {"case": case}
    if op == "net":
        s["net"] = B.Bireal18(_net_params(g, case["stem"] == "module"))
        s["net"].workspace(case["N"])
        s["images"] = torch.randn((case["N"], 3, 224, 224), device="cuda", generator=g)
        return s
    N, C = case["N"], case["C"]
    if op == "pack":
        s["x"] = _activations(g, N, C, case["H"], case["W"], case["layout"])
        return s
    O, k = case["O"], case.get("k", 3)
    s["w"] = B.pack_weights(_weights(g, O, C, k))
    s["scale"], s["shift"] = B.bn_fold(*_bn(g, O))
    if case.get("engine") == "tensor":
        s["wt"] = B.TcWeights(s["w"], C)
    if op == "layer":
        s["x"] = _activations(g, N, C, case["H"], case["W"], case["layout"])
    elif op == "block":
        HW = case["HW"]
        OHW = _out(HW, 3, case["stride"], 1)
        s["a"] = B.pack(_activations(g, N, C, HW, HW, "NHWC"), B.NHWC)
        s["residual"] = torch.randn((N, OHW, OHW, O), device="cuda", generator=g)
    else:
        HW = case["HW"]
        s["x_host"] = _activations(g, N, C, HW, HW, "NCHW").cpu().pin_memory()
        s["out_host"] = torch.empty((N, HW, HW, O), dtype=torch.int32, pin_memory=True)
        s["bits_host"] = torch.empty((N, HW, HW, (O + 63) // 64), dtype=torch.int64, pin_memory=True)
        nbytes = B.binary_layer_host_workspace_bytes(N, C, HW, HW, O, k, k, (1, 1), (k // 2, k // 2), -1)
        s["workspace"] = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    return s


# ---- one pass ---------------------------------------------------------------------------------------------------------
def run(s):
    c = s["case"]
    op = c["op"]
    if op == "net":
        return B.bireal18_forward_stem_module(s["net"], s["images"]) if c["stem"] == "module" else s["net"].forward(s["images"])
    if op == "pack":
        return B.pack(s["x"], B.NCHW if c["layout"] == "NCHW" else B.NHWC)
    if op == "layer":
        geom = ((c["stride"], c["stride"]), (c["pad"], c["pad"]), c["pad_value"])
        a = B.pack(s["x"], B.NCHW if c["layout"] == "NCHW" else B.NHWC)
        if c["engine"] == "tensor":
            return (B.tc_bconv2d(a, s["wt"], *geom) if c["out"] == "int32" else
                    B.tc_bconv2d_bn_sign_pack(a, s["wt"], s["scale"], s["shift"], *geom))
        return (B.bconv2d(a, c["C"], s["w"], *geom) if c["out"] == "int32" else
                B.bconv2d_bn_sign_pack(a, c["C"], s["w"], s["scale"], s["shift"], *geom))
    if op == "block":
        geom = ((c["stride"], c["stride"]), (1, 1), -1)
        if c["engine"] == "tensor":
            return B.tc_bconv2d_bn_add_sign_pack(s["a"], s["wt"], s["scale"], s["shift"], s["residual"], *geom)
        return B.bconv2d_bn_add_sign_pack(s["a"], c["C"], s["w"], s["scale"], s["shift"], s["residual"], *geom)
    pad = c["k"] // 2
    B.binary_layer_host(s["x_host"], s["w"], s["workspace"], (1, 1), (pad, pad), -1, s["scale"], s["shift"],
                        out_host=s["out_host"], bits_host=s["bits_host"])
    return s["out_host"], s["bits_host"]


# ---- what a pass cannot do without ------------------------------------------------------------------------------------
def _words(C):
    return (C + 63) // 64


def work(case):
    """Each input read once, each output written once; a +-1 or fp32 multiply-add counts 2."""
    op, N = case["op"], case["N"]
    if op == "net":
        stem = 112 * 112 * 64 * 147 if case["stem"] == "conv7" else 112 * 112 * (32 * 27 + 16 * 32) + 56 * 56 * (32 * 144 + 64 * 64)
        macs, weight_bytes, C = stem, 64 * 147 * 4 if case["stem"] == "conv7" else (32 * 27 + 512 + 32 * 144 + 4096) * 4, 64
        for b in range(16):
            O, HW = STAGE_C[b // 4], STAGE_HW[b // 4]
            macs += HW * HW * O * C * 9
            weight_bytes += O * C * 9 // 8 + O * 8
            if C != O:
                macs += HW * HW * O * C
                weight_bytes += O * C * 4
            C = O
        macs += 512 * 1000
        return {"bytes": N * (3 * 224 * 224 + 1000) * 4 + weight_bytes + 1000 * 513 * 4, "flops": 2 * N * macs}
    C = case["C"]
    H, W = case.get("H", case.get("HW")), case.get("W", case.get("HW"))
    if op == "pack":
        return {"bytes": N * H * W * (4 * C + 8 * _words(C)), "flops": 0}
    O, k, stride = case["O"], case.get("k", 3), case.get("stride", 1)
    pad = k // 2
    pixels = N * _out(H, k, stride, pad) * _out(W, k, stride, pad)
    nbytes = O * k * k * _words(C) * 8
    if op == "layer":
        nbytes += N * H * W * C * 4 + pixels * (4 * O if case["out"] == "int32" else 8 * _words(O))
    elif op == "block":
        nbytes += N * H * W * _words(C) * 8 + pixels * (8 * O + 8 * _words(O))
    else:
        nbytes += N * H * W * C * 4 + pixels * (4 * O + 8 * _words(O))
    return {"bytes": nbytes, "flops": 2 * pixels * O * C * k * k}


def tolerance(case):
    """Packed words and integer sums are exact.  The fp32 values are single IEEE-rounded operations in the order that the
    library's interface fixes (the next layer takes their sign), so they are the same bits in every correct implementation."""
    return "exact"
