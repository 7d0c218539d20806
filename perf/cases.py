"""The work this framework is used for, as measurable cases.

A case is one call a user's program makes through the public entry points (`paper_2206_07446_b200.binding` and
`.harness`): a whole cold inference, a warm or weights-resident inference, the weight transformation of a model or of
one layer, or the execution of one convolution.  Model shapes are those of the repository's configurations
(ResNet-18/50-, MobileNetV2- and VGG-16-shaped stacks) at a resolution `res`; weights are He-normal, model inputs
uniform in [-1, 1], layer inputs non-negative like the output of a ReLU, batch 1 throughout.

`kernels` names how a model's layers run: "gemm" = 1x1 / im2col GEMM and depthwise kernels, "wino2" / "wino4" / "wino6"
= the same with every 3x3 stride-1 layer on Winograd F(m x m, 3 x 3).
"""
import math

import torch

from paper_2206_07446_b200 import binding as nb
from paper_2206_07446_b200.harness import Model, dev_bytes

MATH = {"fp32": nb.MATH_FP32, "tf32": nb.MATH_TF32, "bf16": nb.MATH_BF16}
VARIANT = {name: i for i, name in enumerate(nb.VARIANT_NAMES)}
WINO_M = {nb.VAR_WINO_F2: 2, nb.VAR_WINO_F4: 4, nb.VAR_WINO_F6: 6}


def listed():
    return [
        # The headline: one cold inference, raw weights from pinned host memory, transformed and executed.
        {"name": "cold_resnet50_224", "op": "cold", "net": "resnet50", "res": 224, "kernels": "gemm", "math": "tf32"},
        # The same of a mobile network: few bytes over the link, many small layers.
        {"name": "cold_mobilenetv2_224", "op": "cold", "net": "mobilenetv2", "res": 224, "kernels": "gemm", "math": "tf32"},
        # The inferences after a cold one in continuous mode: weights prepared, image in, result out.
        {"name": "warm_resnet50_224", "op": "warm", "net": "resnet50", "res": 224, "kernels": "gemm", "math": "tf32"},
        # The same of a mobile network at its usual smaller resolution (odd 5 x 5 grids at the end).
        {"name": "warm_mobilenetv2_160", "op": "warm", "net": "mobilenetv2", "res": 160, "kernels": "gemm", "math": "tf32"},
        # Transformation and execution with the raw weights already in device memory, staged three layers deep.
        {"name": "resident_resnet18_224", "op": "resident", "net": "resnet18", "res": 224, "kernels": "wino4", "math": "tf32"},
        # The decision stage: all post-transform weights of a model, written out once.
        {"name": "transform_all_resnet50", "op": "transform_all", "net": "resnet50", "res": 224, "kernels": "wino6", "math": "tf32"},
        # One small layer's weight transformation: a call that is all latency.
        {"name": "transform_64x64_pack_bf16", "op": "transform", "C": 64, "K": 64, "R": 3, "variant": "im2col", "math": "bf16"},
        # Single convolutions.  The first configuration's layer, ...
        {"name": "conv_3x3_64_56", "op": "conv", "C": 64, "K": 64, "R": 3, "stride": 1, "H": 56, "W": 56,
         "variant": "im2col", "math": "tf32", "bias": False, "residual": False},
        # ... a large VGG-shaped one in bf16, ...
        {"name": "conv_3x3_256_56_bf16", "op": "conv", "C": 256, "K": 256, "R": 3, "stride": 1, "H": 56, "W": 56,
         "variant": "im2col", "math": "bf16", "bias": True, "residual": False},
        # ... a MobileNetV2-shaped 1x1 on a 7 x 7 grid, ...
        {"name": "conv_1x1_320_7", "op": "conv", "C": 320, "K": 1280, "R": 1, "stride": 1, "H": 7, "W": 7,
         "variant": "gemm1x1", "math": "tf32", "bias": True, "residual": False},
        # ... a ragged grid on Winograd F(4x4, 3x3), ...
        {"name": "conv_wino4_ragged", "op": "conv", "C": 96, "K": 160, "R": 3, "stride": 1, "H": 45, "W": 61,
         "variant": "wino_f4", "math": "tf32", "bias": True, "residual": True},
        # ... and a strided one in full fp32, straight from the raw weights.
        {"name": "conv_direct_fp32_s2", "op": "conv", "C": 64, "K": 128, "R": 3, "stride": 2, "H": 56, "W": 56,
         "variant": "direct", "math": "fp32", "bias": False, "residual": False},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Channel counts as networks have them: mostly multiples of 8, some of 32, a few odd."""
    c = _log_int(rng, lo, hi)
    step = rng.choice((1, 8, 8, 32, 32))
    return max(lo, (c + step - 1) // step * step)


MAX_CONV_FLOPS = 3.7e9                                   # of the largest listed convolution
MAX_DIRECT_FLOPS = 0.6e9


def draw(rng):
    op = rng.choice(("cold", "warm", "warm", "resident", "transform_all", "transform", "conv", "conv", "conv", "conv"))
    if op in ("cold", "warm", "resident", "transform_all"):
        net = rng.choice(("resnet50", "mobilenetv2", "resnet18", "vgg16"))
        kernels = "gemm" if op in ("cold", "warm") or net == "mobilenetv2" else rng.choice(("gemm", "wino4", "wino6", "wino2"))
        prec = rng.choice(("tf32", "tf32", "bf16")) if kernels in ("gemm", "wino2") else "tf32"
        return {"op": op, "net": net, "res": _log_int(rng, 96, 224), "kernels": kernels, "math": prec}
    if op == "transform":
        variant = rng.choice(("im2col", "gemm1x1", "wino_f2", "wino_f4", "wino_f6"))
        prec = "tf32" if variant in ("wino_f4", "wino_f6") else rng.choice(("tf32", "bf16"))
        return {"op": op, "C": _channels(rng, 16, 1024), "K": _channels(rng, 16, 1024), "R": 1 if variant == "gemm1x1" else 3,
                "variant": variant, "math": prec}
    variant = rng.choice(("im2col", "im2col", "gemm1x1", "gemm1x1", "wino_f2", "wino_f4", "wino_f6", "direct"))
    prec = "fp32" if variant == "direct" else "tf32" if variant in ("wino_f4", "wino_f6") else rng.choice(("tf32", "tf32", "bf16"))
    R = 1 if variant == "gemm1x1" else 3
    stride = 1 if variant.startswith("wino") else rng.choice((1, 1, 1, 2))
    limit = MAX_DIRECT_FLOPS if variant == "direct" else MAX_CONV_FLOPS
    while True:
        H = _log_int(rng, 7, 224)
        W = H if rng.random() < 0.6 else max(7, min(224, int(H * rng.uniform(0.6, 1.6))))
        c = {"op": "conv", "C": _channels(rng, 16, 1024), "K": _channels(rng, 16, 1024), "R": R, "stride": stride, "H": H, "W": W,
             "variant": variant, "math": prec, "bias": rng.random() < 0.5, "residual": rng.random() < 0.3}
        if work(c)["flops"] <= limit:
            return c


# ---- model shapes ------------------------------------------------------------------------------

def _layer(C, K, R, stride, pad, H, W, in0=-1, in1=-1, act=1, groups=1, bias=0, op=nb.OP_CONV):
    return dict(op=op, C=C, K=K, R=R, S=R, stride=stride, pad=pad, groups=groups, H=H, W=W, in0=in0, in1=in1, act=act,
                has_bias=bias)


def _out(L):
    return (L["H"] + 2 * L["pad"] - L["R"]) // L["stride"] + 1, (L["W"] + 2 * L["pad"] - L["S"]) // L["stride"] + 1


class _Stack:
    """A layer list under construction; shapes follow from the producers."""

    def __init__(self, res):
        self.layers, self.shape = [], {-1: (3, res, res)}

    def add(self, src, K, R, stride=1, pad=None, act=1, depthwise=False, residual=-1, op=nb.OP_CONV):
        C, H, W = self.shape[src]
        L = _layer(C, K, R, stride, R // 2 if pad is None else pad, H, W, src, residual, act, C if depthwise else 1, 0, op)
        self.layers.append(L)
        self.shape[len(self.layers) - 1] = (K,) + _out(L)
        return len(self.layers) - 1

    def pool(self, src, R, stride, pad):
        return self.add(src, self.shape[src][0], R, stride, pad, 0, op=nb.OP_MAXPOOL)


def _network(net, res):
    n = _Stack(res)
    if net in ("resnet18", "resnet50"):
        deep = net == "resnet50"
        x = n.pool(n.add(-1, 64, 7, 2), 3, 2, 1)
        width = 64
        for stage, (mid, blocks) in enumerate(zip((64, 128, 256, 512), (3, 4, 6, 3) if deep else (2, 2, 2, 2))):
            out = 4 * mid if deep else mid
            for b in range(blocks):
                s = 2 if stage and b == 0 else 1
                if deep:
                    y = n.add(n.add(x, mid, 1), mid, 3, s)
                else:
                    y = n.add(x, mid, 3, s)
                skip = x if s == 1 and width == out else n.add(x, out, 1, s, act=0)
                x = n.add(y, out, 1 if deep else 3, residual=skip)
                width = out
    elif net == "vgg16":
        x = -1
        for stage, (K, convs) in enumerate(((64, 2), (128, 2), (256, 3), (512, 3), (512, 3))):
            for _ in range(convs):
                x = n.add(x, K, 3)
            if stage < 4:
                x = n.pool(x, 2, 2, 0)
    else:
        x = n.add(-1, 32, 3, 2, act=2)
        width = 32
        for expand, K, blocks, stride in ((1, 16, 1, 1), (6, 24, 2, 2), (6, 32, 3, 2), (6, 64, 4, 2), (6, 96, 3, 1), (6, 160, 3, 2),
                                          (6, 320, 1, 1)):
            for b in range(blocks):
                s = stride if b == 0 else 1
                h = n.add(x, width * expand, 1, act=2) if expand > 1 else x
                h = n.add(h, width * expand, 3, s, act=2, depthwise=True)
                x = n.add(h, K, 1, act=0, residual=x if s == 1 and width == K else -1)
                width = K
        n.add(x, 1280, 1, act=2)
    return n.layers


def _layers(case):
    if "net" in case:
        return _network(case["net"], case["res"])
    H, W = case.get("H", 14), case.get("W", 14)                        # a weight transformation does not depend on the grid
    return [_layer(case["C"], case["K"], case["R"], case.get("stride", 1), case["R"] // 2, H, W, bias=int(case.get("bias", False)))]


def _choices(case, layers):
    """(variant, math, raw weights) per layer; None for pools."""
    out = []
    for L in layers:
        if L["op"] != nb.OP_CONV:
            out.append(None)
        elif "variant" in case:
            out.append((VARIANT[case["variant"]], MATH[case["math"]], nb.ARM_RAW))
        elif L["groups"] > 1:
            out.append((nb.VAR_DEPTHWISE, nb.MATH_FP32, nb.ARM_RAW))
        else:
            wino = {"wino2": nb.VAR_WINO_F2, "wino4": nb.VAR_WINO_F4, "wino6": nb.VAR_WINO_F6}.get(case["kernels"])
            v = nb.VAR_GEMM1X1 if L["R"] == 1 else wino if wino and L["R"] == 3 and L["stride"] == 1 else nb.VAR_IM2COL
            out.append((v, MATH[case["math"]], nb.ARM_RAW))
    return out


def _weights(layers, gen):
    """He-normal OIHW weights of every layer as one blob on the GPU: (float32 tensor, byte offsets of weights and biases)."""
    w_off, b_off, pos = [], [], 0
    for L in layers:
        conv = L["op"] == nb.OP_CONV
        w_off.append(4 * pos)
        pos += -(-(L["K"] * L["C"] // L["groups"] * L["R"] * L["S"]) // 64) * 64 if conv else 0
        b_off.append(4 * pos)
        pos += -(-L["K"] // 64) * 64 if conv and L["has_bias"] else 0
    blob = torch.randn(max(64, pos), generator=gen, device="cuda")
    for L, w, b in zip(layers, w_off, b_off):
        if L["op"] == nb.OP_CONV:
            cg = L["C"] // L["groups"]
            blob[w // 4:w // 4 + L["K"] * cg * L["R"] * L["S"]] *= math.sqrt(2.0 / (cg * L["R"] * L["S"]))
            if L["has_bias"]:
                blob[b // 4:b // 4 + L["K"]] *= 0.1
    return blob, w_off, b_off


# ---- one pass ----------------------------------------------------------------------------------

def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    layers = _layers(case)
    choices = _choices(case, layers)
    blob, w_off, b_off = _weights(layers, gen)
    s = {"op": case["op"], "stream": torch.cuda.current_stream()}
    if case["op"] in ("cold", "warm", "resident"):
        # a cold inference happens once per process and is enqueued call by call; repeated ones replay a recorded graph
        m = Model(layers, blob.cpu().numpy().view("uint8"), w_off, b_off, use_graphs=0 if case["op"] == "cold" else 1)
        x = torch.rand(m.h_input.shape, generator=gen, device="cuda") * 2 - 1
        m.h_input.copy_(x)
        s["model"], s["choices"] = m, nb.choices_array(m.plan, choices)
        s["depth"] = 3 if case["op"] == "resident" else 0
        m.ensure_arena(choices, s["depth"])
        if case["op"] == "warm":
            m.cold_run_continuous(m.h_input.numpy(), choices, choices)
        elif case["op"] == "resident":
            m.to_device()
            m.d_input.copy_(x)
        torch.cuda.synchronize()
        return s
    s["plan"], s["w"], s["w_bytes"] = nb.nnv_plan_create(layers, w_off, b_off), blob, 4 * blob.numel()
    if case["op"] == "transform_all":
        s["choices"] = nb.choices_array(s["plan"], choices)
        _, total = nb.nnv_transformed_layout(s["plan"], s["choices"])
        s["out"] = dev_bytes(total, fill=0)
        s["result"] = s["out"].view(torch.bfloat16 if case["math"] == "bf16" else torch.float32)
        return s
    v, m, _ = choices[0]
    s["kernel"] = (v, m)
    direct = v == nb.VAR_DIRECT
    nbytes = 0 if direct else nb.nnv_transformed_bytes(s["plan"], 0, v, m)
    wt = blob if direct else dev_bytes(nbytes, fill=0)
    if case["op"] == "transform":
        s["out"] = wt
        s["result"] = wt[:nbytes].view(torch.bfloat16 if m == nb.MATH_BF16 else torch.float32)
        return s
    L = layers[0]
    if not direct:
        nb.nnv_transform_weights(s["plan"], 0, v, m, blob, wt, s["stream"])
    oh, ow = _out(L)
    s["wt"], s["bias"] = wt, blob[b_off[0] // 4:] if L["has_bias"] else None
    s["x"] = torch.randn((L["H"], L["W"], L["C"]), generator=gen, device="cuda").relu_()
    s["addend"] = torch.randn((oh, ow, L["K"]), generator=gen, device="cuda") if case["residual"] else None
    s["y"] = torch.empty((oh, ow, L["K"]), device="cuda")
    s["ws_bytes"] = nb.nnv_exec_workspace_bytes(s["plan"], 0, v, m)
    s["ws"] = dev_bytes(s["ws_bytes"], fill=None) if s["ws_bytes"] else None
    return s


def run(s):
    op = s["op"]
    if op == "conv":
        nb.nnv_conv_exec(s["plan"], 0, s["kernel"][0], s["kernel"][1], s["x"], s["addend"], s["wt"], s["bias"], s["y"], s["ws"],
                         s["ws_bytes"], s["stream"])
        return s["y"]
    if op == "transform":
        nb.nnv_transform_weights(s["plan"], 0, s["kernel"][0], s["kernel"][1], s["w"], s["out"], s["stream"])
        return s["result"]
    if op == "transform_all":
        nb.nnv_transform_all(s["plan"], s["choices"], s["w"], s["w_bytes"], s["out"], s["out"].numel(), s["stream"])
        return s["result"]
    m = s["model"]
    if op == "cold":
        nb.nnv_cold_run(m.plan, s["choices"], m.h_weights, m.w_bytes, None, 0, m.h_input, m.h_output, m.arena, m.arena.numel(),
                        m.streams[0], m.streams[1], m.streams[2], s["depth"])
        return m.h_output
    if op == "warm":
        nb.nnv_warm_run(m.plan, s["choices"], m.d_warm, m.warm_bytes, m.w_bytes, m.h_input, m.h_output, m.arena, m.arena.numel(),
                        m.streams[1], m.streams[2])
        return m.h_output
    nb.nnv_resident_run(m.plan, s["choices"], m.d_weights, m.w_bytes, None, 0, m.d_input, m.d_output, m.arena, m.arena.numel(),
                        m.streams[1], m.streams[2], s["depth"])
    return m.d_output


# ---- what a pass cannot do without ---------------------------------------------------------------

def _packed_bytes(L, choice):
    """Bytes of a layer's weights as its kernel reads them."""
    v, m, _ = choice
    n, es = L["K"] * (L["C"] // L["groups"]), 2 if m == nb.MATH_BF16 else 4
    return n * es * ((WINO_M[v] + 2) ** 2 if v in WINO_M else L["R"] * L["S"])


def work(case):
    layers = _layers(case)
    choices = _choices(case, layers)
    raw = prepared = reads = flops = 0
    for L, c in zip(layers, choices):
        oh, ow = _out(L)
        if L["op"] != nb.OP_CONV:
            continue
        raw += 4 * (L["K"] * (L["C"] // L["groups"]) * L["R"] * L["S"] + (L["K"] if L["has_bias"] else 0))
        prepared += _packed_bytes(L, c) if c[0] not in (nb.VAR_DIRECT, nb.VAR_DEPTHWISE) else 0
        reads += _packed_bytes(L, c) + (4 * L["K"] if L["has_bias"] else 0)
        if c[0] in WINO_M:
            t = WINO_M[c[0]]
            flops += 2 * (t + 2) ** 2 * -(-oh // t) * -(-ow // t) * L["K"] * L["C"]
        else:
            flops += 2 * oh * ow * L["K"] * (L["C"] // L["groups"]) * L["R"] * L["S"]
    if case["op"] in ("transform", "transform_all"):
        return {"bytes": raw + prepared, "flops": 0}
    first, last = layers[0], layers[-1]
    oh, ow = _out(last)
    io = 4 * (first["C"] * first["H"] * first["W"] + last["K"] * oh * ow * (2 if case.get("residual") else 1))
    # cold and resident passes read the raw weights; warm passes and single layers the prepared ones
    return {"bytes": io + (reads if case["op"] in ("warm", "conv") else raw), "flops": flops}


def tolerance(case):
    """One TF32 pass is good to 1e-3, one bf16 pass to 1e-2, fp32 sums to 1e-5 (the accuracy classes of the kernels); F(4x4)
    and F(6x6) multiply error-compensated operands.  A model chains its layers' errors."""
    if case["op"] in ("transform", "transform_all"):
        wino = case.get("kernels", case.get("variant", "")).startswith("wino")
        if not wino:
            return "exact"                                             # a repack moves and rounds, it does not add
        return {"rel": 3e-3, "max": 1e-2} if case["math"] == "bf16" else {"rel": 1e-5, "max": 1e-3}
    if "net" in case:
        return {"rel": 1e-2 if case["math"] == "tf32" else 2.5e-2, "max": 0.5}
    if case["math"] == "fp32":
        return {"rel": 1e-5}
    if case["variant"] in ("wino_f4", "wino_f6"):
        return {"rel": 2e-4}
    return {"rel": 1e-3 if case["math"] == "tf32" else 1e-2}
