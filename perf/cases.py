"""The workloads whose speed is measured: what a program that runs 8-bit CNN inference has the library do.

Five kinds of work, each through the public entry points of `paper_1805_08691_b200`:

  conv        one quantized convolution (`q8_conv2d`), as a host that walks its own layer list calls it: from the
              single-image layer, where launch latency is all there is, to layers that fill the tensor cores;
              channel counts that are no multiple of 16, strides, 1xN filters, residual sums, fp32 outputs and
              per-channel multipliers included
  bottleneck  `pipeline.Bottleneck`: 1x1, 3x3, 1x1 + identity residual, the building block of the residual networks
  network     `network.QuantNetwork.forward` on a batch of fp32 images (ResNet-50, Inception-v3, SSD-300 with the
              L2-normalised conv4_3), either called directly or captured once in a CUDA graph and replayed
  quantize    the calibration and conversion of an activation tensor: running max-abs, Eq. (Q), Eq. (D)
  detect      `q8_detection_output` on the head tensors of a detector

All outputs are integer arithmetic or single IEEE operations in a fixed order, so every case compares bit for bit.
"""
import math
from types import SimpleNamespace

import torch
import torch.nn.functional as F

from paper_1805_08691_b200 import binding as q8
from paper_1805_08691_b200 import network, pipeline

DEV = "cuda"


# ------------------------------------------------------------------------------------------------ the cases
def _conv(name, N, H, W, C, K, R, S, stride=1, pad_h=0, pad_w=0, dil=1, x="u8", y="u8", res="", relu=True, per_channel=False):
    return {"name": name, "kind": "conv", "N": N, "H": H, "W": W, "C": C, "K": K, "R": R, "S": S, "stride": stride,
            "pad_h": pad_h, "pad_w": pad_w, "dil": dil, "x": x, "y": y, "res": res, "relu": relu, "per_channel": per_channel}


def _bottleneck(name, N, HW, C):
    return {"name": name, "kind": "bottleneck", "N": N, "HW": HW, "C": C}


def _network(name, net, N, graph, streams=4, per_channel=False):
    return {"name": name, "kind": "network", "net": net, "N": N, "graph": graph, "streams": streams, "per_channel": per_channel}


def listed():
    return [
        # a single layer on one image: the latency of one call
        _conv("conv_3x3_14x14_c64_b1", 1, 14, 14, 64, 64, 3, 3, pad_h=1, pad_w=1),
        # the first layer of a network on images as they come, three channels, not padded to 16
        _conv("conv_first_3x3s2_c3_b8", 8, 299, 299, 3, 32, 3, 3, stride=2, x="s8"),
        # a factorized filter of an Inception module: odd map, channel count between the powers of two
        _conv("conv_1x7_17x17_c160_b64", 64, 17, 17, 160, 160, 1, 7, pad_w=3),
        # a VGG layer at detection size: bound by the tensor cores
        _conv("conv_3x3_75x75_c256_b32", 32, 75, 75, 256, 256, 3, 3, pad_h=1, pad_w=1),
        # the residual block of the early and of the late stages
        _bottleneck("bottleneck_56x56_c256_b32", 32, 56, 256),
        _bottleneck("bottleneck_14x14_c1024_b64", 64, 14, 1024),
        # serving at throughput: one captured graph per batch; latency of a single image: direct calls
        _network("resnet50_b64_graph", "resnet50", 64, True),
        _network("resnet50_b1", "resnet50", 1, False),
        _network("inception_v3_b64", "inception_v3", 64, False),
        # detection: the largest network; heads are returned dequantized
        _network("ssd300_b32", "ssd300", 32, False),
        # calibration and conversion of a stage-2 activation tensor
        {"name": "quantize_56x56_c256_b64", "kind": "quantize", "N": 64, "H": 56, "W": 56, "C": 256, "type": "u8"},
        # post-processing of 32 images, 8732 boxes, 21 classes
        {"name": "detect_b32", "kind": "detect", "N": 32, "cells": 38, "classes": 21},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["conv"] * 5 + ["bottleneck"] * 2 + ["network"] * 3 + ["quantize"] + ["detect"])
    if kind == "conv":
        while True:
            R, S, pad_h, pad_w = rng.choice([(1, 1, 0, 0), (1, 1, 0, 0), (3, 3, 1, 1), (3, 3, 1, 1), (3, 3, 0, 0), (1, 7, 0, 3),
                                             (7, 1, 3, 0), (5, 5, 2, 2), (7, 7, 3, 3)])
            aligned = rng.random() < 0.85
            C = 16 * _log(rng, 1, 96) if aligned else rng.choice([3, 3, _log(rng, 5, 200)])
            K = 16 * _log(rng, 1, 64) if rng.random() < 0.8 else _log(rng, 8, 500)
            side = _log(rng, 4, 224)
            N = _log(rng, 1, 64)
            stride, dil = (2 if rng.random() < 0.2 else 1), 1
            if (R, S) == (3, 3) and rng.random() < 0.1:
                dil, pad_h, pad_w, stride = 2, 2, 2, 1
            c = _conv("", N, side, max(4, side + rng.randint(-2, 2)), C, K, R, S, stride, pad_h, pad_w, dil,
                      x="s8" if C == 3 or rng.random() < 0.15 else "u8", y=rng.choice(["u8"] * 6 + ["s8", "f32"]),
                      res="u8" if rng.random() < 0.25 else "", relu=rng.random() < 0.8, per_channel=rng.random() < 0.2)
            del c["name"]
            P, Q = _extent(c)
            # up to the work of the largest listed layer; layers off the 16-channel grid up to that of a stem layer
            macs = N * P * Q * K * R * S * C
            if P >= 1 and Q >= 1 and 1e5 <= macs <= (1.1e11 if C % 16 == 0 else 5e8) and R * S * C <= 16384 \
                    and N * side * side * C <= 1.5e8 and N * P * Q * K <= 1.5e8:
                return c
    if kind == "bottleneck":
        C, HW = rng.choice([(256, 56), (512, 28), (1024, 14), (2048, 7)])
        c = _bottleneck("", _log(rng, 1, 64), max(4, HW + rng.randint(-3, 8)), C)
        del c["name"]
        return c
    if kind == "network":
        net = rng.choice(["resnet50", "inception_v3", "ssd300"])
        c = _network("", net, _log(rng, 1, {"resnet50": 64, "inception_v3": 56, "ssd300": 28}[net]), rng.random() < 0.4,
                     rng.choice([1, 2, 4, 4, 4]), rng.random() < 0.2)
        del c["name"]
        return c
    if kind == "quantize":
        return {"kind": "quantize", "N": _log(rng, 1, 64), "H": _log(rng, 7, 56), "W": _log(rng, 7, 56), "C": _log(rng, 3, 256),
                "type": rng.choice(["u8", "s8"])}
    return {"kind": "detect", "N": _log(rng, 1, 32), "cells": rng.randint(10, 38), "classes": rng.randint(3, 21)}


# ------------------------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV)


def _he(g, K, R, S, C):
    return _randn(g, K, R, S, C) * math.sqrt(2.0 / (R * S * C))


def _codes(g, shape, kind):
    """Quantized activations: ReLU(N(0,1)) as u8 or N(0,1) as s8, factor 5 / 255 or 5 / 127."""
    x = _randn(g, *shape)
    if kind == "s8":
        return q8.q8_quantize(x, 5.0 / 127, q8.Q8_S8)
    return q8.q8_quantize(x.relu_(), 5.0 / 255, q8.Q8_U8)


def _extent(c):
    P = (c["H"] + 2 * c["pad_h"] - c["dil"] * (c["R"] - 1) - 1) // c["stride"] + 1
    Q = (c["W"] + 2 * c["pad_w"] - c["dil"] * (c["S"] - 1) - 1) // c["stride"] + 1
    return P, Q


TYPES = {"u8": q8.Q8_U8, "s8": q8.Q8_S8, "f32": q8.Q8_F32}
FACTOR = {"u8": 5.0 / 255, "s8": 5.0 / 127, "f32": 1.0}


def _prepare_conv(c, g):
    N, H, W, C, K = (c[k] for k in "NHWCK")
    P, Q = _extent(c)
    w, b = _he(g, K, c["R"], c["S"], C), _randn(g, K) * 0.01
    qc = pipeline.prepare_conv(w, b, (N, H, W, C), FACTOR[c["x"]], FACTOR[c["y"]], TYPES[c["x"]], TYPES[c["y"]], c["relu"],
                               (c["stride"],) * 2, (c["pad_h"], c["pad_w"]), (c["dil"],) * 2,
                               FACTOR[c["res"]] if c["res"] else None, TYPES[c["res"] or "u8"], per_channel=c["per_channel"])
    nbytes = q8.q8_conv2d_workspace_bytes(qc.desc)
    return SimpleNamespace(qc=qc, x=_codes(g, (N, H, W, C), c["x"]), res=_codes(g, (N, P, Q, K), c["res"]) if c["res"] else None,
                           out=torch.empty((N, P, Q, K), dtype=q8.TORCH_DTYPES[TYPES[c["y"]]], device=DEV),
                           ws=torch.empty(nbytes, dtype=torch.uint8, device=DEV) if nbytes else None)


def _run_conv(s):
    qc = s.qc
    return q8.q8_conv2d(qc.desc, s.x, qc.w_q, qc.b_q, qc.scale, s.res, qc.res_scale, s.out, s.ws)


def _prepare_bottleneck(c, g):
    N, HW, C = c["N"], c["HW"], c["C"]
    mid = C // 4
    folded = [(_he(g, k, r, r, ci), _randn(g, k) * 0.1) for k, r, ci in ((mid, 1, C), (mid, 3, mid), (C, 1, mid))]
    block = pipeline.Bottleneck(folded, {"x": 5.0, "a": 5.0, "b": 5.0, "c": 5.0}, (N, HW, HW, C))
    return SimpleNamespace(block=block, x=_codes(g, (N, HW, HW, C), "u8"), out=torch.empty((N, HW, HW, C), dtype=torch.uint8, device=DEV))


# ------------------------------------------------------------------------------------------------ networks
class _Layers(list):
    """A layer list as QuantNetwork takes it, with seeded weights (He-normal, BN as in a trained network's ranges)."""

    def __init__(self, g):
        super().__init__()
        self.g = g
        self.params = {}

    def add(self, name, op, src, **kw):
        d = dict(name=name, op=op, src=list(src), conv=None, residual=None, f32_out=False, k=(1, 1), stride=(1, 1), pad=(0, 0),
                 ceil_mode=False, gamma=None, eps=1e-10)
        d.update(kw)
        self.append(SimpleNamespace(**d))
        return name

    def conv(self, name, src, C, K, R=1, S=None, stride=1, pad=(0, 0), dil=1, relu=True, bn=True, residual=None, f32_out=False):
        S = R if S is None else S
        pad = (pad, pad) if isinstance(pad, int) else pad
        spec = SimpleNamespace(C=C, K=K, R=R, S=S, stride=(stride, stride), pad=pad, dil=(dil, dil), relu=relu)
        self.params[name] = (_he(self.g, K, R, S, C), bn)
        return self.add(name, "conv", [src], conv=spec, residual=residual, f32_out=f32_out)

    def pool(self, name, src, op, k, stride=1, pad=0, ceil_mode=False):
        return self.add(name, op, [src], k=(k, k), stride=(stride, stride), pad=(pad, pad), ceil_mode=ceil_mode)

    def folded(self):
        g, out = self.g, {}
        for L in self:
            if L.op != "conv":
                continue
            w, bn = self.params[L.name]
            K = L.conv.K
            if bn:
                u = torch.rand((2, K), generator=g, device=DEV) + 0.5
                m = _randn(g, 2, K) * 0.1
                out[L.name] = q8.q8_fold_bn(w, None, u[0].contiguous(), m[0].contiguous(), m[1].contiguous(), u[1].contiguous())
            else:
                out[L.name] = (w, _randn(g, K) * 0.01)
        return out


def _resnet50(g):
    L = _Layers(g)
    L.conv("conv1", "input", 3, 64, 7, stride=2, pad=3)
    x, c = L.pool("pool1", "conv1", "maxpool", 3, 2, 1), 64
    for stage, (blocks, mid) in enumerate(zip((3, 4, 6, 3), (64, 128, 256, 512)), start=2):
        for b in range(blocks):
            t, st, short = f"res{stage}{'abcdef'[b]}", (2 if b == 0 and stage > 2 else 1), x
            if b == 0:
                short = L.conv(t + "_branch1", x, c, 4 * mid, stride=st, relu=False)
            y = L.conv(t + "_branch2a", x, c, mid, stride=st)
            y = L.conv(t + "_branch2b", y, mid, mid, 3, pad=1)
            x, c = L.conv(t + "_branch2c", y, mid, 4 * mid, residual=short), 4 * mid
    L.pool("pool5", x, "avgpool", 7)
    L.conv("fc1000", "pool5", 2048, 1000, relu=False, bn=False, f32_out=True)
    return L, 224


def _inception_v3(g):
    L = _Layers(g)

    def chain(x, c, *steps):  # steps: (name, K, R, S, stride, pad)
        for name, K, R, S, st, pad in steps:
            x, c = L.conv(name, x, c, K, R, S, st, pad), K
        return x

    x = chain("input", 3, ("conv1", 32, 3, 3, 2, 0), ("conv2", 32, 3, 3, 1, 0), ("conv3", 64, 3, 3, 1, 1))
    x = L.pool("pool1", x, "maxpool", 3, 2)
    x = chain(x, 64, ("conv4", 80, 1, 1, 1, 0), ("conv5", 192, 3, 3, 1, 0))
    x, c = L.pool("pool2", x, "maxpool", 3, 2), 192
    for i, pf in enumerate((32, 64, 64)):
        t = f"m{i}_"
        br = [chain(x, c, (t + "1x1", 64, 1, 1, 1, 0)),
              chain(x, c, (t + "5x5r", 48, 1, 1, 1, 0), (t + "5x5", 64, 5, 5, 1, 2)),
              chain(x, c, (t + "3x3r", 64, 1, 1, 1, 0), (t + "3x3a", 96, 3, 3, 1, 1), (t + "3x3b", 96, 3, 3, 1, 1)),
              chain(L.pool(t + "pool", x, "avgpool", 3, 1, 1), c, (t + "proj", pf, 1, 1, 1, 0))]
        x, c = L.add(f"m{i}", "concat", br), 224 + pf
    br = [chain(x, c, ("m3_3x3", 384, 3, 3, 2, 0)),
          chain(x, c, ("m3_r", 64, 1, 1, 1, 0), ("m3_a", 96, 3, 3, 1, 1), ("m3_b", 96, 3, 3, 2, 0)), L.pool("m3_pool", x, "maxpool", 3, 2)]
    x, c = L.add("m3", "concat", br), 480 + c
    for i, k in enumerate((128, 160, 160, 192), start=4):
        t = f"m{i}_"
        br = [chain(x, c, (t + "1x1", 192, 1, 1, 1, 0)),
              chain(x, c, (t + "7r", k, 1, 1, 1, 0), (t + "1x7", k, 1, 7, 1, (0, 3)), (t + "7x1", 192, 7, 1, 1, (3, 0))),
              chain(x, c, (t + "dr", k, 1, 1, 1, 0), (t + "d7x1a", k, 7, 1, 1, (3, 0)), (t + "d1x7a", k, 1, 7, 1, (0, 3)),
                    (t + "d7x1b", k, 7, 1, 1, (3, 0)), (t + "d1x7b", 192, 1, 7, 1, (0, 3))),
              chain(L.pool(t + "pool", x, "avgpool", 3, 1, 1), c, (t + "proj", 192, 1, 1, 1, 0))]
        x, c = L.add(f"m{i}", "concat", br), 768
    br = [chain(x, c, ("m8_r", 192, 1, 1, 1, 0), ("m8_3x3", 320, 3, 3, 2, 0)),
          chain(x, c, ("m8_7r", 192, 1, 1, 1, 0), ("m8_1x7", 192, 1, 7, 1, (0, 3)), ("m8_7x1", 192, 7, 1, 1, (3, 0)),
                ("m8_7x3", 192, 3, 3, 2, 0)), L.pool("m8_pool", x, "maxpool", 3, 2)]
    x, c = L.add("m8", "concat", br), 1280
    for i in (9, 10):
        t = f"m{i}_"
        r = chain(x, c, (t + "r", 384, 1, 1, 1, 0))
        b2 = L.add(t + "b2", "concat", [chain(r, 384, (t + "1x3", 384, 1, 3, 1, (0, 1))), chain(r, 384, (t + "3x1", 384, 3, 1, 1, (1, 0)))])
        r = chain(x, c, (t + "dr", 448, 1, 1, 1, 0), (t + "d3x3", 384, 3, 3, 1, 1))
        b3 = L.add(t + "b3", "concat", [chain(r, 384, (t + "d1x3", 384, 1, 3, 1, (0, 1))), chain(r, 384, (t + "d3x1", 384, 3, 1, 1, (1, 0)))])
        br = [chain(x, c, (t + "1x1", 320, 1, 1, 1, 0)), b2, b3,
              chain(L.pool(t + "pool", x, "avgpool", 3, 1, 1), c, (t + "proj", 192, 1, 1, 1, 0))]
        x, c = L.add(f"m{i}", "concat", br), 2048
    L.pool("pool3", x, "avgpool", 8)
    L.conv("fc", "pool3", 2048, 1000, relu=False, bn=False, f32_out=True)
    return L, 299


def _ssd300(g):
    L = _Layers(g)
    x, c = "input", 3
    for stage, (n, k) in enumerate(((2, 64), (2, 128), (3, 256), (3, 512), (3, 512)), start=1):
        for i in range(1, n + 1):
            x, c = L.conv(f"conv{stage}_{i}", x, c, k, 3, pad=1, bn=False), k
        if stage < 5:
            x = L.pool(f"pool{stage}", x, "maxpool", 2, 2, ceil_mode=stage == 3)
    L.add("norm4", "l2norm", ["conv4_3"], gamma=(torch.rand(512, generator=g, device=DEV) * 10 + 15).cpu().numpy())
    x = L.pool("pool5", x, "maxpool", 3, 1, 1)
    heads = [("norm4", 512, 4)]
    x = L.conv("fc6", x, 512, 1024, 3, pad=6, dil=6, bn=False)
    x = L.conv("fc7", x, 1024, 1024, bn=False)
    heads.append((x, 1024, 6))
    c = 1024
    for i, (mid, k, st, pad, boxes) in enumerate(((256, 512, 2, 1, 6), (128, 256, 2, 1, 6), (128, 256, 1, 0, 4), (128, 256, 1, 0, 4)), start=6):
        x = L.conv(f"conv{i}_1", x, c, mid, bn=False)
        x, c = L.conv(f"conv{i}_2", x, mid, k, 3, stride=st, pad=pad, bn=False), k
        heads.append((x, c, boxes))
    for src, c, boxes in heads:
        L.conv(src + "_loc", src, c, boxes * 4, 3, pad=1, relu=False, bn=False, f32_out=True)
        L.conv(src + "_conf", src, c, boxes * 21, 3, pad=1, relu=False, bn=False, f32_out=True)
    return L, 300


NETS = {"resnet50": _resnet50, "inception_v3": _inception_v3, "ssd300": _ssd300}


def _calibrate(layers, folded, x):
    """Max-abs of every tensor of the FP32 network on a batch of images (NHWC), as the deployment step collects them."""
    out, seen = {"input": x.permute(0, 3, 1, 2)}, {"input": x}
    with torch.no_grad(), torch.backends.cudnn.flags(enabled=True, benchmark=False, deterministic=True, allow_tf32=False):
        for L in layers:
            a = out[L.src[0]]
            if L.op == "conv":
                w, b = folded[L.name]
                y = F.conv2d(a, w.permute(0, 3, 1, 2), b, L.conv.stride, L.conv.pad, L.conv.dil)
                if L.residual is not None:
                    seen[L.name + ":pre"] = y
                    y = y + out[L.residual]
                if L.conv.relu:
                    y = y.relu()
            elif L.op == "maxpool":
                y = F.max_pool2d(a, L.k, L.stride, L.pad, ceil_mode=L.ceil_mode)
            elif L.op == "avgpool":
                y = F.avg_pool2d(a, L.k, L.stride, L.pad)
            elif L.op == "concat":
                y = torch.cat([out[s] for s in L.src], 1)
            else:
                y = a / (a.square().sum(1, keepdim=True) + L.eps).sqrt() * torch.from_numpy(L.gamma).to(DEV).view(1, -1, 1, 1)
            out[L.name] = seen[L.name] = y
    cal = pipeline.Calibrator(sorted(seen))
    for name, t in seen.items():
        cal.observe(name, t.contiguous())
    return cal.maxima()


def _prepare_network(c, g):
    layers, hw = NETS[c["net"]](g)
    folded = layers.folded()
    maxima = _calibrate(layers, folded, _randn(g, 1, hw, hw, 3))
    x = _randn(g, c["N"], hw, hw, 3)
    net = network.QuantNetwork(layers, folded, maxima, x.shape, streams=c["streams"], per_channel=c["per_channel"])
    s = SimpleNamespace(net=net, x=x, outs=[L.name for L in layers if L.f32_out], graph=None, result=None)
    if c["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            net.forward(x)
        torch.cuda.current_stream().wait_stream(side)
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            s.result = net.forward(x)
    return s


def _run_network(s):
    if s.graph is not None:
        s.graph.replay()
        out = s.result
    else:
        out = s.net.forward(s.x)
    return {name: out[name] for name in s.outs}


# ------------------------------------------------------------------------------------------------ conversion, detection
def _prepare_quantize(c, g):
    x = _randn(g, c["N"], c["H"], c["W"], c["C"])
    if c["type"] == "u8":
        x.relu_()
    return SimpleNamespace(x=x, type=TYPES[c["type"]], q=FACTOR[c["type"]], slot=torch.zeros(1, device=DEV),
                           z=torch.empty(x.shape, dtype=q8.TORCH_DTYPES[TYPES[c["type"]]], device=DEV), r=torch.empty_like(x))


def _run_quantize(s):
    q8.q8_calibrate_maxabs(s.x, s.slot)
    q8.q8_quantize(s.x, s.q, s.type, out=s.z)
    q8.q8_dequantize(s.z, s.q, out=s.r)
    return s.slot, s.z, s.r


BOXES = ((1.0, 4), (0.5, 6), (0.26, 6), (0.13, 6), (0.08, 4), (0.03, 4))  # source maps: side relative to the first, boxes per cell


def _maps(c):
    return [(max(1, int(math.ceil(c["cells"] * f))), b) for f, b in BOXES]


def _prepare_detect(c, g):
    """Head outputs with the structure of a trained detector's: offsets N(0,1); logits N(0,1), background raised by 8,
    2 % of the boxes given one class raised by 4 to 9."""
    N, classes = c["N"], c["classes"]
    sources, priors = [], []
    for i, (side, boxes) in enumerate(_maps(c)):
        n = side * side * boxes
        loc = _randn(g, N, side, side, boxes * 4)
        conf = _randn(g, N, n, classes)
        conf[..., 0] += 8.0
        hot = torch.rand((N, n, 1), generator=g, device=DEV) < 0.02
        cls = torch.randint(1, classes, (N, n, 1), generator=g, device=DEV)
        conf.scatter_add_(2, cls, hot * (torch.rand((N, n, 1), generator=g, device=DEV) * 5 + 4))
        sources.append((loc, conf.view(N, side, side, boxes * classes), boxes))
        ys, xs = torch.meshgrid(torch.arange(side, device=DEV), torch.arange(side, device=DEV), indexing="ij")
        centre = torch.stack([(xs + 0.5) / side, (ys + 0.5) / side], -1).view(-1, 1, 2).expand(-1, boxes, 2)
        ratio = torch.tensor([1.0, 1.2, 2.0, 0.5, 3.0, 1.0 / 3][:boxes], device=DEV).sqrt()
        size = (0.1 + 0.16 * i) * torch.stack([ratio, 1.0 / ratio], -1).view(1, boxes, 2).expand(side * side, boxes, 2)
        priors.append(torch.cat([centre, size], -1).reshape(-1, 4))
    priors = torch.cat(priors).contiguous()
    nbytes = q8.q8_detection_output_workspace_bytes(N, priors.shape[0], classes, 0, 400, 200)
    return SimpleNamespace(sources=sources, priors=priors, classes=classes, ws=torch.empty(nbytes, dtype=torch.uint8, device=DEV),
                           out=torch.empty((N, 200, 6), device=DEV), counts=torch.empty(N, dtype=torch.int32, device=DEV))


def _run_detect(s):
    return q8.q8_detection_output(s.sources, s.priors, (0.1, 0.1, 0.2, 0.2), s.classes, workspace=s.ws, out=s.out, counts=s.counts)


# ------------------------------------------------------------------------------------------------ interface
PREPARE = {"conv": _prepare_conv, "bottleneck": _prepare_bottleneck, "network": _prepare_network, "quantize": _prepare_quantize,
           "detect": _prepare_detect}


def prepare(case, seed):
    s = PREPARE[case["kind"]](case, _gen(seed))
    s.kind = case["kind"]
    return s


def run(state):
    if state.kind == "conv":
        return _run_conv(state)
    if state.kind == "bottleneck":
        return state.block(state.x, out=state.out)
    if state.kind == "network":
        return _run_network(state)
    if state.kind == "quantize":
        return _run_quantize(state)
    return _run_detect(state)


#: (multiply-accumulates of one image, bytes of 8-bit weights and biases, bytes of fp32 outputs of one image)
NET_WORK = {"resnet50": (3857973248, 25.6e6, 4000), "inception_v3": (5713216096, 23.8e6, 4000), "ssd300": (31373537792, 26.4e6, 8732 * 25 * 4)}
NET_SIDE = {"resnet50": 224, "inception_v3": 299, "ssd300": 300}
SIZE = {"u8": 1, "s8": 1, "f32": 4, "": 0}


def work(case):
    k = case["kind"]
    if k == "conv":
        P, Q = _extent(case)
        N, C, K, taps = case["N"], case["C"], case["K"], case["R"] * case["S"]
        out = N * P * Q * K
        return {"bytes": N * case["H"] * case["W"] * C + K * taps * C + 4 * K + out * (SIZE[case["y"]] + SIZE[case["res"]]),
                "flops": 2.0 * out * taps * C}
    if k == "bottleneck":
        M, C = case["N"] * case["HW"] ** 2, case["C"]
        params = C * C // 4 * 2 + 9 * C * C // 16
        return {"bytes": 2 * M * C + params, "flops": 2.0 * M * params}
    if k == "network":
        macs, params, out = NET_WORK[case["net"]]
        return {"bytes": case["N"] * (12 * NET_SIDE[case["net"]] ** 2 + out) + params, "flops": 2.0 * macs * case["N"]}
    if k == "quantize":
        n = case["N"] * case["H"] * case["W"] * case["C"]
        return {"bytes": 9 * n, "flops": 3.0 * n}   # fp32 in once, codes and fp32 out once
    boxes = sum(side * side * b for side, b in _maps(case))
    return {"bytes": case["N"] * (boxes * 4 * (4 + case["classes"]) + 200 * 24) + 16 * boxes, "flops": 10.0 * case["N"] * boxes * case["classes"]}


def tolerance(case):
    return "exact"
