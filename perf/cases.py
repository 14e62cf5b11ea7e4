"""Performance cases of the routine-selecting inference library.

A program that uses the library builds a net, tunes it (profile, select a
path), keeps the tuned handle and then runs it on input after input, replayed
as a CUDA graph on its own stream; or it calls the adapt conversion on its
own.  The cases follow that: single convolutions, the residual, inverted
residual and squeeze-and-excite blocks that the nets are made of, two whole
nets, and adapts, in fp32, fp16, bf16 and qint8, at batch 1 to 32.

The path of a case is tuned once per process and kept (`_paths`): every state
of the case is a net of its own with its own weights and buffers on that
path, as a program keeps a tuned plan and loads it for the next net.
"""
from __future__ import annotations

import json
import math

import torch

import paper_2110_06037_gb300 as sn

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16, "qi8": torch.int8}
SIZE = {"f32": 4, "f16": 2, "bf16": 2, "qi8": 1}

# scale of the qint8 input blob: unit normal values fill +-4 of the code range
Q_IN = 4.0 / 127.0

_paths = {}
_stream = None


def listed():
    return [
        # the headline workload: a whole ResNet-50 at batch 32, throughput serving
        {"name": "resnet50_b32", "kind": "net", "arch": "resnet50", "dtype": "bf16", "n": 32, "hw": 224},
        # interactive use: a whole MobileNetV2 at batch 1, where latency and launches count
        {"name": "mobilenetv2_b1", "kind": "net", "arch": "mobilenet_v2", "dtype": "f16", "n": 1, "hw": 224},
        # the smallest call: one stage-3 bottleneck of ResNet-50 at batch 1
        {"name": "bottleneck_b1", "kind": "bottleneck", "dtype": "f16", "n": 1, "hw": 14, "c": 1024, "mid": 256,
         "out": 1024, "stride": 1},
        # the same kind of block at serving batch, stage 2
        {"name": "bottleneck_b32", "kind": "bottleneck", "dtype": "bf16", "n": 32, "hw": 28, "c": 512, "mid": 128,
         "out": 512, "stride": 1},
        # the first block of a stage: stride 2 and a projection shortcut
        {"name": "bottleneck_down_b8", "kind": "bottleneck", "dtype": "f16", "n": 8, "hw": 56, "c": 256, "mid": 128,
         "out": 512, "stride": 2},
        # fp32 inference, the natural type of an unquantised net
        {"name": "bottleneck_f32_b8", "kind": "bottleneck", "dtype": "f32", "n": 8, "hw": 28, "c": 512, "mid": 128,
         "out": 512, "stride": 1},
        # the largest layer of the single-layer convolution sweep
        {"name": "conv_512_b32", "kind": "conv", "dtype": "f16", "n": 32, "hw": 56, "c": 512, "k": 512, "ks": 3,
         "stride": 1, "layout": "nhwc"},
        # an odd map, odd batch, large kernel and stride 2 in the layout that importers produce
        {"name": "conv_ragged", "kind": "conv", "dtype": "f16", "n": 5, "hw": 35, "c": 72, "k": 120, "ks": 5,
         "stride": 2, "layout": "nchw"},
        # a MobileNetV2 block at serving batch: pointwise, depthwise, pointwise, residual
        {"name": "inverted_b32", "kind": "inverted", "dtype": "f16", "n": 32, "hw": 28, "c": 32, "exp": 192, "ks": 3,
         "act": "relu6", "se": False},
        # a MobileNetV3 block: 5x5 depthwise and squeeze-and-excite
        {"name": "inverted_se_b8", "kind": "inverted", "dtype": "bf16", "n": 8, "hw": 28, "c": 40, "exp": 120, "ks": 5,
         "act": "hswish", "se": True},
        # the same kind of block tuned over the qint8 schemas, as a quantised mobile net runs it
        {"name": "inverted_q8_b8", "kind": "inverted", "dtype": "qi8", "n": 8, "hw": 14, "c": 112, "exp": 672, "ks": 3,
         "act": "hswish", "se": True},
        # feeding an fp32 NCHW producer's maps to an fp16 NHWC consumer
        {"name": "adapt_f32_f16", "kind": "adapt", "from": "f32", "from_layout": "nchw", "to": "f16",
         "to_layout": "nhwc", "n": 32, "c": 256, "h": 28, "w": 28},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mult8(rng, lo, hi):
    return max(8, _log_int(rng, lo, hi) // 8 * 8)


def draw(rng):
    kind = rng.choice(["net", "bottleneck", "bottleneck", "conv", "conv", "inverted", "inverted", "adapt"])
    while True:
        if kind == "net":
            # (a random-weight MobileNetV2 in bf16 is already 3e-2 off fp64: no tolerance could be stated for it)
            arch, dtype = rng.choice([("resnet50", "bf16"), ("resnet50", "f16"), ("mobilenet_v2", "f16")])
            case = {"kind": kind, "arch": arch, "dtype": dtype, "n": _log_int(rng, 1, 24),
                    "hw": rng.choice([128, 160, 192, 224])}
        elif kind == "bottleneck":
            mid = _mult8(rng, 64, 256)
            dtype = rng.choice(["f16", "bf16", "f32"])
            stride = rng.choice([1, 1, 2])
            c = 4 * mid if stride == 1 else 2 * mid
            case = {"kind": kind, "dtype": dtype, "n": _log_int(rng, 1, 8 if dtype == "f32" else 32),
                    "hw": rng.randint(7, 56), "c": c, "mid": mid, "out": 4 * mid, "stride": stride}
        elif kind == "conv":
            # channel counts are multiples of 8 in most layers; the others are a net's first and last ones
            c, k = _mult8(rng, 32, 512), _mult8(rng, 32, 512)
            odd = rng.random() < 0.2
            case = {"kind": kind, "dtype": rng.choice(["f16", "bf16"]),
                    "n": _log_int(rng, 1, 4 if odd else 32), "hw": rng.randint(7, 56),
                    "c": _log_int(rng, 3, 64) if odd else c, "k": _log_int(rng, 10, 128) if odd else k,
                    "ks": rng.choice([1, 3, 3, 5]), "stride": rng.choice([1, 2]),
                    "layout": rng.choice(["nhwc", "nchw"])}
        elif kind == "inverted":
            c = _mult8(rng, 16, 160)
            case = {"kind": kind, "dtype": rng.choice(["f16", "bf16", "qi8"]), "n": _log_int(rng, 1, 32),
                    "hw": rng.randint(7, 56), "c": c, "exp": c * rng.choice([3, 4, 6]), "ks": rng.choice([3, 3, 5]),
                    "act": rng.choice(["relu6", "hswish"]), "se": rng.random() < 0.5}
        else:
            a, b = rng.choice([("f32", "f16"), ("f32", "bf16"), ("f16", "f16"), ("bf16", "bf16"), ("f16", "f32"),
                               ("bf16", "f32"), ("f32", "f32")])
            lay = ["nchw", "nhwc"]
            rng.shuffle(lay)
            case = {"kind": kind, "from": a, "from_layout": lay[0], "to": b, "to_layout": lay[1],
                    "n": _log_int(rng, 1, 32), "c": _log_int(rng, 3, 512), "h": rng.randint(7, 112),
                    "w": rng.randint(7, 112)}
        w = work(case)
        # below the largest listed convolution, whose tuning alone takes seconds
        if w["flops"] <= 100e9 and w["bytes"] <= 400e6:
            return case


# ------------------------------------------------------------------ the nets

def _conv(layers, src, c, k, ks, stride, act, gain=1.0, groups=1):
    layers.append({"type": "conv2" if groups == 1 else "dwconv2", "inputs": [src], "gain": gain,
                   "params": dict(c_in=c, c_out=k, kh=ks, kw=ks, sh=stride, sw=stride, ph=ks // 2, pw=ks // 2, dh=1,
                                  dw=1, groups=groups, act=act)})
    return len(layers) - 1


def _push(layers, type_, inputs, **params):
    layers.append({"type": type_, "inputs": list(inputs), "params": params})
    return len(layers) - 1


def _bottleneck(layers, src, c, mid, out, stride):
    """1x1, 3x3, 1x1 and the shortcut; the last scale of a residual branch is small, as a trained net's is."""
    t = _conv(layers, src, c, mid, 1, 1, "relu")
    t = _conv(layers, t, mid, mid, 3, stride, "relu")
    t = _conv(layers, t, mid, out, 1, 1, "none", gain=0.25)
    if stride != 1 or c != out:
        src = _push_projection(layers, src, c, out, stride)
    return _push(layers, "add", [src, t], act="relu")


def _push_projection(layers, src, c, out, stride):
    layers.append({"type": "conv2", "inputs": [src], "gain": 1.0,
                   "params": dict(c_in=c, c_out=out, kh=1, kw=1, sh=stride, sw=stride, ph=0, pw=0, dh=1, dw=1,
                                  groups=1, act="none")})
    return len(layers) - 1


def _inverted(layers, src, c, exp, out, ks, stride, act, se):
    t = _conv(layers, src, c, exp, 1, 1, act) if exp != c else src
    t = _conv(layers, t, exp, exp, ks, stride, act, groups=exp)
    if se:
        red = max(8, exp // 4 // 8 * 8)
        s = _push(layers, "gap", [t])
        s = _push(layers, "dense", [s], in_features=exp, out_features=red, act="relu")
        s = _push(layers, "dense", [s], in_features=red, out_features=exp, act="hsigmoid")
        t = _push(layers, "mul", [t, s], act="none")
    t = _conv(layers, t, exp, out, 1, 1, "none")
    return _push(layers, "add", [src, t], act="none") if stride == 1 and c == out else t


def _net(case):
    """(layers, logical NCHW input shape) of a case."""
    layers = []
    if case["kind"] == "conv":
        _conv(layers, -1, case["c"], case["k"], case["ks"], case["stride"], "relu")
    elif case["kind"] == "bottleneck":
        _bottleneck(layers, -1, case["c"], case["mid"], case["out"], case["stride"])
    elif case["kind"] == "inverted":
        _inverted(layers, -1, case["c"], case["exp"], case["c"], case["ks"], 1, case["act"], case["se"])
    elif case["arch"] == "resnet50":
        t = _conv(layers, -1, 3, 64, 7, 2, "relu")
        t = _push(layers, "maxpool", [t], kh=3, kw=3, sh=2, sw=2, ph=1, pw=1)
        c = 64
        for mid, out, n, s in [(64, 256, 3, 1), (128, 512, 4, 2), (256, 1024, 6, 2), (512, 2048, 3, 2)]:
            for i in range(n):
                t = _bottleneck(layers, t, c, mid, out, s if i == 0 else 1)
                c = out
        t = _push(layers, "gap", [t])
        _push(layers, "dense", [t], in_features=2048, out_features=1000, act="none")
    else:
        t = _conv(layers, -1, 3, 32, 3, 2, "relu6")
        c = 32
        for e, out, n, s in [(1, 16, 1, 1), (6, 24, 2, 2), (6, 32, 3, 2), (6, 64, 4, 2), (6, 96, 3, 1),
                             (6, 160, 3, 2), (6, 320, 1, 1)]:
            for i in range(n):
                t = _inverted(layers, t, c, c * e, out, 3, s if i == 0 else 1, "relu6", False)
                c = out
        t = _conv(layers, t, c, 1280, 1, 1, "relu6")
        t = _push(layers, "gap", [t])
        _push(layers, "dense", [t], in_features=1280, out_features=1000, act="none")
    c = 3 if case["kind"] == "net" else case["c"]
    return layers, (case["n"], c, case["hw"], case["hw"])


def _shapes(layers, in_shape):
    out = []
    for l in layers:
        n, c, h, w = in_shape if l["inputs"][0] < 0 else out[l["inputs"][0]]
        p = l["params"]
        if l["type"] in ("conv2", "dwconv2", "maxpool"):
            h = (h + 2 * p["ph"] - p["kh"]) // p["sh"] + 1
            w = (w + 2 * p["pw"] - p["kw"]) // p["sw"] + 1
            c = p.get("c_out", c)
        elif l["type"] == "gap":
            h = w = 1
        elif l["type"] == "dense":
            c = p["out_features"]
        out.append((n, c, h, w))
    return out


def _weight_shape(l):
    p = l["params"]
    if l["type"] in ("conv2", "dwconv2"):
        return p["c_out"], p["c_in"] // p["groups"], p["kh"], p["kw"]
    if l["type"] == "dense":
        return p["out_features"], p["in_features"]
    return None


def _materialise(case, seed):
    """(layers with weights on the GPU, input) of a seed: unit normal input, He-normal weights, biases of
    standard deviation 0.1, all values of the case's own type (fp32 for qint8, whose weights are quantised
    by the library)."""
    layers, shape = _net(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float32 if case["dtype"] == "qi8" else DTYPES[case["dtype"]]
    x = torch.randn(shape, generator=gen, device="cuda")
    if case["dtype"] == "qi8":
        x = torch.clamp(torch.round(x / Q_IN), -127, 127).to(torch.int8)
    else:
        x = x.to(dt)
    for l in layers:
        ws = _weight_shape(l)
        if ws is None:
            continue
        w = torch.randn(ws, generator=gen, device="cuda") * (l.get("gain", 1.0) * math.sqrt(2.0 / math.prod(ws[1:])))
        l["w"] = w.to(dt).float()
        l["b"] = torch.randn(ws[0], generator=gen, device="cuda") * 0.1
    return layers, x


def _act(v, act):
    if act == "relu":
        return v.clamp(min=0)
    if act == "relu6":
        return v.clamp(0, 6)
    if act in ("hswish", "hsigmoid"):
        t = (v + 3).clamp(0, 6) / 6
        return v * t if act == "hswish" else t
    return v


def _forward(layers, x, keep_all=False):
    """The net in the type of x: convolutions as one matrix product per tap."""
    blobs = []
    for l in layers:
        ins = [x if j < 0 else blobs[j] for j in l["inputs"]]
        v, p = ins[0], l["params"]
        if l["type"] in ("conv2", "dwconv2"):
            w = l["w"].to(x.dtype)
            v = torch.nn.functional.pad(v, (p["pw"], p["pw"], p["ph"], p["ph"]))
            h = (v.shape[2] - p["kh"]) // p["sh"] + 1
            q = (v.shape[3] - p["kw"]) // p["sw"] + 1
            acc = None
            for r in range(p["kh"]):
                for s in range(p["kw"]):
                    t = v[:, :, r:r + (h - 1) * p["sh"] + 1:p["sh"], s:s + (q - 1) * p["sw"] + 1:p["sw"]]
                    if l["type"] == "conv2":
                        t = torch.matmul(w[:, :, r, s], t.reshape(t.shape[0], t.shape[1], h * q))
                    else:
                        t = (t * w[:, 0, r, s].view(1, -1, 1, 1)).reshape(t.shape[0], t.shape[1], h * q)
                    acc = t if acc is None else acc.add_(t)
            v = (acc + l["b"].to(x.dtype).view(1, -1, 1)).view(v.shape[0], -1, h, q)
        elif l["type"] == "maxpool":
            v = torch.nn.functional.pad(v, (p["pw"], p["pw"], p["ph"], p["ph"]), value=float("-inf"))
            v = v.unfold(2, p["kh"], p["sh"]).unfold(3, p["kw"], p["sw"]).amax((-1, -2))
        elif l["type"] == "gap":
            v = v.mean((2, 3), keepdim=True)
        elif l["type"] == "dense":
            v = (v.flatten(1) @ l["w"].to(x.dtype).T + l["b"].to(x.dtype)).view(v.shape[0], -1, 1, 1)
        elif l["type"] == "add":
            v = v + ins[1]
        elif l["type"] == "mul":
            v = v * ins[1]
        blobs.append(_act(v, p.get("act", "none")))
    return blobs if keep_all else blobs[-1]


def _io_schema(case):
    # nets take the importers' NCHW; blocks and layers sit inside a net that runs in NHWC unless they say otherwise
    return case["dtype"], "nchw" if case["kind"] == "net" else case.get("layout", "nhwc")


# ---------------------------------------------------------------- the cases

def _adapt_input(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (case["n"], case["c"], case["h"], case["w"])
    x = torch.randn(sn.storage_shape(shape, case["from_layout"]), generator=gen, device="cuda")
    return shape, x.to(DTYPES[case["from"]])


def prepare(case, seed):
    global _stream
    if case["kind"] == "adapt":
        shape, x = _adapt_input(case, seed)
        out = torch.empty(sn.storage_shape(shape, case["to_layout"]), dtype=DTYPES[case["to"]], device="cuda")
        return {"x": x, "out": out, "shape": shape, "from": (case["from"], case["from_layout"]),
                "to": (case["to"], case["to_layout"])}
    if _stream is None:
        _stream = torch.cuda.Stream()
    layers, x = _materialise(case, seed)
    scales = None
    if case["dtype"] == "qi8":  # calibration: the largest value of each blob on this input
        scales = [float(v.abs().max()) / 127.0 or 1.0 for v in _forward(layers, x.float() * Q_IN, keep_all=True)]
    desc = [dict(type=l["type"], inputs=l["inputs"], params=l["params"],
                 weight=l["w"].cpu().numpy() if "w" in l else None, bias=l["b"].cpu().numpy() if "b" in l else None)
            for l in layers]
    shape = tuple(x.shape)
    io = _io_schema(case)
    lam = [(case["dtype"], "nchw"), (case["dtype"], "nhwc")]
    if io[1] == "nhwc":
        x = x.permute(0, 2, 3, 1).contiguous()
    torch.cuda.synchronize()
    g = sn.build_graph(desc, shape, io, io, lam, fuse=True)
    if scales is not None:
        g.set_qscale(-1, Q_IN)
        for old, new in enumerate(g.fused_ids):
            if new >= 0:
                g.set_qscale(new, scales[old])
    key = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    if key not in _paths:
        # as many launches a candidate as tuning in a few seconds allows: the slowest routines are ~1000 times
        # slower than the fastest
        iters = int(max(2, min(20, 4e10 / work(case)["flops"])))
        if case["kind"] == "net":
            iters = 10
        g.profile(warmup=2 if iters > 2 else 1, iters=iters, topk=3, passes=7, stream=_stream)
        _, _, cands = g.select_path(sn.SN_SELECT_DPRS)
        _paths[key] = [int(c) for c in cands]
    else:
        g.set_path(_paths[key])
    g.set_option(sn.SN_OPT_CUDA_GRAPH, 1)
    g.plan_stats(stream=_stream)  # the weights in the path's formats and the buffers
    return {"g": g, "x": x, "out": g.new_output(), "stream": _stream}


def run(state):
    if "g" in state:
        return state["g"].run(state["x"], state["out"], stream=state["stream"])
    return sn.convert(state["x"], state["from"], state["to"], state["shape"], out=state["out"])


def work(case):
    if case["kind"] == "adapt":
        n = case["n"] * case["c"] * case["h"] * case["w"]
        return {"bytes": n * (SIZE[case["from"]] + SIZE[case["to"]]), "flops": 0}
    layers, shape = _net(case)
    shapes = _shapes(layers, shape)
    es = SIZE[case["dtype"]]
    nbytes = es * (math.prod(shape) + math.prod(shapes[-1]))
    flops = 0
    for l, s in zip(layers, shapes):
        ws = _weight_shape(l)
        if ws is None:
            flops += math.prod(s)
            continue
        nbytes += es * math.prod(ws) + 4 * ws[0]
        flops += 2 * math.prod(s) * math.prod(ws[1:])
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """About four times the error against fp64 measured on these cases."""
    if case["kind"] == "adapt" or case["dtype"] == "qi8":
        return "exact"  # adapts round to nearest even, qint8 routines are defined to the bit
    if case["dtype"] == "f32":
        return {"rel": 1e-5}  # measured 4e-7 to 1.2e-6 on blocks whose 3x3 layer runs as Winograd
    if case["kind"] == "net":
        # measured 4.4e-3 (MobileNetV2, fp16) and 2.5e-3 (ResNet-50, bf16)
        return {"rel": 0.017 if case["arch"] == "mobilenet_v2" else 0.01}
    # measured 2.1e-4 to 3.9e-4 (fp16), 1.8e-3 to 2.6e-3 (bf16)
    return {"rel": 0.002 if case["dtype"] == "f16" else 0.01}


def exact(case, seed):
    if case["kind"] == "adapt":
        _, x = _adapt_input(case, seed)
        if case["from_layout"] != case["to_layout"]:
            x = x.permute(0, 2, 3, 1) if case["to_layout"] == "nhwc" else x.permute(0, 3, 1, 2)
        return x.double().contiguous()
    if case["dtype"] == "qi8":
        return None  # codes: whole numbers, which are compared as such
    layers, x = _materialise(case, seed)
    y = _forward(layers, x.double())
    return y.permute(0, 2, 3, 1).contiguous() if _io_schema(case)[1] == "nhwc" else y.contiguous()
