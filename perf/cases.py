"""What is measured: pattern-pruned 3x3 convolutions through the package's public entry points.

A user packs a layer once (``api.pp_pack(...).bind()``), keeps one workspace for the layers of the
network (``api.workspace_for``) and output buffers, and then calls ``layer.conv`` per layer and
batch.  The cases are single layers of the repository's workloads (VGG-16, ResNet-50's 3x3
convolutions, MobileNet-V2's depthwise layers, the single-layer sweep), odd sizes between them, and
the whole VGG-16 stack at batch 1 (latency) and 32 (throughput).  ``draw`` gives further single
layers of the same ranges: 3 to 512 channels, maps of 7 to 224, batches of 1 to 256, strides 1 and
2, connectivity keep 0.25 to 1, fp32 and fp16, with and without the fused 2x2 max-pool, dense and
depthwise.

Inputs are what the layers meet: ReLU(N(0, 1)) activations (N(0, 1) for 3-channel images) and
He-normal weights, bias N(0, 0.1^2), every layer with bias and ReLU.
"""
from __future__ import annotations

import math

import torch
import torch.nn.functional as F

from paper_2003_06513_gb300 import api

# --------------------------------------------------------------------------------------- cases

LARGEST_FLOP = 2 ** 37     # useful FLOP of a drawn layer, below the whole stack's at batch 32
LARGEST_BYTES = 2 ** 30    # activations of a drawn layer


def _conv(name, cin, cout, h, w, n, keep, dtype="f32", stride=1, pool=False):
    return {"name": name, "kind": "conv", "cin": cin, "cout": cout, "h": h, "w": w, "n": n,
            "keep": keep, "dtype": dtype, "stride": stride, "pool": pool}


def _depthwise(name, c, h, w, n, dtype="f16", stride=1):
    return {"name": name, "kind": "depthwise", "cin": c, "cout": c, "h": h, "w": w, "n": n,
            "keep": 1.0, "dtype": dtype, "stride": stride, "pool": False}


def listed():
    return [
        # the smallest call: one image through one small layer, all launch and latency
        _conv("single_64x32_n1", 64, 64, 32, 32, 1, 0.5),
        # one image through the VGG-16 stack: the latency a serving program sees
        {"name": "vgg16_n1", "kind": "vgg16", "n": 1},
        # the first block's second layer with its pool: the largest maps, few channels
        _conv("vgg2_224_n32_pool", 64, 64, 224, 224, 32, 0.3, pool=True),
        # the middle of the network, ordinary batch
        _conv("vgg6_56_n32", 256, 256, 56, 56, 32, 0.3),
        # late layers: small maps, many channels
        _conv("vgg12_14_n32", 512, 512, 14, 14, 32, 0.3),
        # a ResNet-50 stage head (stride 2)
        _conv("r50_head_28_n64", 256, 256, 28, 28, 64, 0.4, stride=2),
        # ResNet-50's last stage: 7x7 maps, rows of odd length
        _conv("r50_7_n64", 512, 512, 7, 7, 64, 0.4),
        # half precision in the sweep's ranges, a layer with every kernel kept
        _conv("sweep_28_n64_f16", 256, 256, 28, 28, 64, 1.0, dtype="f16"),
        # ragged: channel counts off the group size, an odd map, a small batch
        _conv("ragged_45x61_n5", 90, 150, 45, 61, 5, 0.5),
        # MobileNet-V2 depthwise: large planes, and the smallest planes
        _depthwise("dw_56_n128_f16", 144, 56, 56, 128),
        _depthwise("dw_7_n128_f16", 960, 7, 7, 128),
        # the whole VGG-16 stack at the throughput batch
        {"name": "vgg16_n32", "kind": "vgg16", "n": 32},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        n = _log(rng, 1, 256)
        h = _log(rng, 7, 224)
        w = h if rng.random() < 0.5 else max(7, min(224, int(h * rng.uniform(0.6, 1.6))))
        stride = 2 if rng.random() < 0.25 else 1
        dtype = "f16" if rng.random() < 0.35 else "f32"
        if rng.random() < 0.2:
            c = _log(rng, 32, 960)
            case = _depthwise("", c, h, w, n, dtype, stride)
        else:
            cin = 3 if rng.random() < 0.08 else _log(rng, 16, 512)
            cout = cin if cin > 3 and rng.random() < 0.5 else _log(rng, 16, 512)
            if rng.random() < 0.6:                       # networks use multiples of 16
                cin, cout = cin if cin == 3 else 16 * -(-cin // 16), 16 * -(-cout // 16)
            keep = rng.choice([0.25, 0.3, 0.4, 0.5, 1.0])
            case = _conv("", cin, cout, h, w, n, keep, dtype, stride, stride == 1 and rng.random() < 0.25)
        del case["name"]
        wk = work(case)
        if wk["flops"] <= LARGEST_FLOP and wk["bytes"] <= LARGEST_BYTES:
            return case


# ------------------------------------------------------------------------------------- a layer

_DT = {"f32": torch.float32, "f16": torch.float16}


def _out_hw(case):
    s = case["stride"]
    ho, wo = (case["h"] - 1) // s + 1, (case["w"] - 1) // s + 1
    return (ho // 2, wo // 2) if case["pool"] else (ho, wo)


def _cin_g(case):
    return 1 if case["kind"] == "depthwise" else case["cin"]


def _kept(case):
    k = case["cout"] * _cin_g(case)
    return max(1, min(k, math.floor(case["keep"] * k + 0.5)))


VGG16 = [(3, 64, 224, False), (64, 64, 224, True), (64, 128, 112, False), (128, 128, 112, True),
         (128, 256, 56, False), (256, 256, 56, False), (256, 256, 56, True), (256, 512, 28, False),
         (512, 512, 28, False), (512, 512, 28, True), (512, 512, 14, False), (512, 512, 14, False),
         (512, 512, 14, True)]


def _vgg16_layers(n):
    return [_conv("", ci, co, h, h, n, 1.0 if ci == 3 else 0.3, pool=pool) for ci, co, h, pool in VGG16]


def _weights(case, gen):
    """Host weights and bias of one layer."""
    std = math.sqrt(2.0 / (9 * _cin_g(case)))
    W = torch.randn(case["cout"], _cin_g(case), 3, 3, generator=gen) * std
    return W, torch.randn(case["cout"], generator=gen) * 0.1


def _input(case, seed, relu):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.randn(case["n"], case["cin"], case["h"], case["w"], generator=gen, device="cuda",
                    dtype=_DT[case["dtype"]])
    return x.relu_() if relu else x


def _layers(case):
    return _vgg16_layers(case["n"]) if case["kind"] == "vgg16" else [case]


def prepare(case, seed):
    """Packed and bound layers, biases, the input, one shared workspace and the outputs."""
    gen = torch.Generator().manual_seed(seed)
    specs = _layers(case)
    layers, biases, outs, shapes = [], [], [], []
    for spec in specs:
        W, b = _weights(spec, gen)
        groups = spec["cout"] if spec["kind"] == "depthwise" else 1
        layers.append(api.pp_pack(W.numpy(), None, spec["keep"], groups, spec["stride"]).bind("cuda"))
        biases.append(b.cuda())
        shapes.append((spec["n"], spec["cin"], spec["h"], spec["w"]))
        outs.append(torch.empty((spec["n"], spec["cout"]) + _out_hw(spec), device="cuda",
                                dtype=_DT[spec["dtype"]]))
    pools = [spec["pool"] for spec in specs]
    nbytes = max(lay.workspace_bytes(s, p, _DT[spec["dtype"]])
                 for lay, s, p, spec in zip(layers, shapes, pools, specs))
    ws = torch.empty(nbytes // 4 + 4, device="cuda") if nbytes else None
    x = _input(specs[0], seed, relu=specs[0]["cin"] > 3)
    torch.cuda.synchronize()
    return {"x": x, "layers": layers, "biases": biases, "outs": outs, "pools": pools, "ws": ws}


def run(state):
    """One forward pass: every layer's convolution + bias + ReLU (+ pool), on the current stream."""
    cur = state["x"]
    for lay, b, out, pool in zip(state["layers"], state["biases"], state["outs"], state["pools"]):
        cur = lay.conv(cur, b, True, out=out, workspace=state["ws"], pool2x2=pool)
    return cur


def work(case):
    """Useful FLOP (4 kept weights a kernel) and the bytes of each layer's input, output, kept
    weights with their positions, and bias."""
    nbytes = flops = 0
    for spec in _layers(case):
        es = 4 if spec["dtype"] == "f32" else 2
        ho, wo = (spec["h"] - 1) // spec["stride"] + 1, (spec["w"] - 1) // spec["stride"] + 1
        po, qo = _out_hw(spec)
        flops += 8 * _kept(spec) * spec["n"] * ho * wo
        nbytes += es * spec["n"] * (spec["cin"] * spec["h"] * spec["w"] + spec["cout"] * po * qo)
        nbytes += 17 * _kept(spec) + 4 * spec["cout"]
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- the same in 64 bits

# the default library: centre + 3 of the 4 edge neighbours, centre + an edge and its two corners
PATTERNS = [(3, 4, 5, 7), (1, 4, 5, 7), (1, 3, 4, 7), (1, 3, 4, 5),
            (0, 1, 2, 4), (0, 3, 4, 6), (2, 4, 5, 8), (4, 6, 7, 8)]


def _projected(W, keep):
    """Weights after pattern projection (per kernel the pattern that retains the largest norm) and
    connectivity pruning (the kernels that retain the most), in 64 bits."""
    cout, cin = W.shape[:2]
    k = W.double().reshape(cout * cin, 9)
    score = torch.stack([sum(k[:, t] * k[:, t] for t in p) for p in PATTERNS], 1)
    best = score.argmax(1)
    mask = torch.zeros(len(PATTERNS), 9, dtype=torch.float64)
    for i, p in enumerate(PATTERNS):
        mask[i, list(p)] = 1.0
    kept = max(1, min(k.shape[0], math.floor(keep * k.shape[0] + 0.5)))
    order = torch.argsort(score.max(1).values, descending=True, stable=True)
    alive = torch.zeros(k.shape[0], 1, dtype=torch.float64)
    alive[order[:kept]] = 1.0
    return (k * mask[best] * alive).reshape(cout, cin, 3, 3)


def _conv64(x, W, stride):
    """3x3 convolution, padding 1, as nine shifted products (dense) or F.conv2d (depthwise)."""
    n, cin, h, w = x.shape
    ho, wo = (h - 1) // stride + 1, (w - 1) // stride + 1
    xp = F.pad(x, (1, 1, 1, 1))
    if W.shape[1] == 1 and cin > 1:
        y = torch.zeros(n, cin, ho, wo, dtype=torch.float64, device=x.device)
        for t in range(9):
            dy, dx = divmod(t, 3)
            part = xp[:, :, dy:dy + (ho - 1) * stride + 1:stride, dx:dx + (wo - 1) * stride + 1:stride]
            y += part * W[:, 0, dy, dx].view(1, -1, 1, 1)
        return y
    y = torch.zeros(W.shape[0], n * ho * wo, dtype=torch.float64, device=x.device)
    for t in range(9):
        dy, dx = divmod(t, 3)
        part = xp[:, :, dy:dy + (ho - 1) * stride + 1:stride, dx:dx + (wo - 1) * stride + 1:stride]
        y.addmm_(W[:, :, dy, dx].contiguous(), part.permute(1, 0, 2, 3).reshape(cin, -1))
    return y.view(W.shape[0], n, ho, wo).permute(1, 0, 2, 3)


def exact(case, seed):
    gen = torch.Generator().manual_seed(seed)
    specs = _layers(case)
    cur = None
    params = [_weights(spec, gen) for spec in specs]
    x = _input(specs[0], seed, relu=specs[0]["cin"] > 3)
    out = []
    step = max(1, (1 << 27) // (max(s["cin"] + s["cout"] for s in specs) * specs[0]["h"] * specs[0]["w"]))
    proj = [(_projected(W, spec["keep"]).cuda(), b.double().cuda()) for (W, b), spec in zip(params, specs)]
    for i in range(0, x.shape[0], step):
        cur = x[i:i + step].double()
        for (W, b), spec in zip(proj, specs):
            cur = (_conv64(cur, W, spec["stride"]) + b.view(1, -1, 1, 1)).relu_()
            if spec["pool"]:
                cur = F.max_pool2d(cur, 2)
        out.append(cur)
    return torch.cat(out)


def tolerance(case):
    """About four times the error seen against ``exact``: fp32 sums of up to 2048 products 1e-7 to
    3e-7 of the result, the thirteen-layer stack 1.4e-7, four-product depthwise sums 3e-8; fp16
    outputs 2.1e-4, the root mean square of their rounding."""
    if case["kind"] == "vgg16":
        return {"rel": 1e-6}
    if case["dtype"] == "f16":
        return {"rel": 8e-4}
    return {"rel": 2e-7 if case["kind"] == "depthwise" else 1.2e-6}
