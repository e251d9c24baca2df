"""The work that a user of the library has it do, as measurable cases.

A case is one pass through the C ABI's binding as a program calls it: one layer, the layers of a network one after the
other, a fused block, or a layer whose activations live in host memory.  Shapes follow the layer tables of
``paper_2006_09791_b200.workloads`` and the shape lists of the tests; `draw` varies batch, image size, channels, groups
and filters around them.  All tensors are fp32 (the library has no other type); results follow the variant the library
picks (TF32 tensor cores or FP32).
"""
from __future__ import annotations

import math
import weakref

import torch

from paper_2006_09791_b200 import gconv
from paper_2006_09791_b200.torch_util import attach_workspace


# ---- layers of a case ------------------------------------------------------------------------------------------------
# A layer: (N, C_in, H, W, C_out, (KH, KW), (stride), (pad), (dilation), groups)
def _conv(N, Ci, H, W, Co, k=(3, 3), stride=(1, 1), pad=(1, 1), dil=(1, 1), groups=1):
    return (N, Ci, H, W, Co, k, stride, pad, dil, groups)


def _out_hw(L):
    N, Ci, H, W, Co, k, s, p, d, g = L
    return ((H + 2 * p[0] - d[0] * (k[0] - 1) - 1) // s[0] + 1, (W + 2 * p[1] - d[1] * (k[1] - 1) - 1) // s[1] + 1)


def _half(v):
    """Plane size behind a 3x3 layer with stride 2 and pad 1."""
    return (v - 1) // 2 + 1


def _planes(size):
    """Plane sizes of a five-stage network on size x size images, from size / 2 to size / 32."""
    out = [_half(size)]
    while len(out) < 5:
        out.append(_half(out[-1]))
    return out


def _stack_layers(N, size, C, g):
    """WideResNet-40-2-shaped stack: three stages of six 3x3 layers, channels C / 2C / 4C, stride 2 into stages 2 and 3."""
    a, b, c = size, _half(size), _half(_half(size))
    s2 = (2, 2)
    return ([_conv(N, C, a, a, C, groups=g)] * 6 + [_conv(N, C, a, a, 2 * C, stride=s2, groups=g)] +
            [_conv(N, 2 * C, b, b, 2 * C, groups=g)] * 5 + [_conv(N, 2 * C, b, b, 4 * C, stride=s2, groups=g)] +
            [_conv(N, 4 * C, c, c, 4 * C, groups=g)] * 5)


def _resnet_layers(N, size, C, g):
    """ResNet-34-shaped 3x3 layers: channels C ... 8C at size / 4 ... size / 32, stride 2 between the stages."""
    out = []
    for i, hw in enumerate(_planes(size)[1:]):
        c = C << i
        out.append(_conv(N, c, hw, hw, c, groups=g))
        if i < 3:
            out.append(_conv(N, c, hw, hw, 2 * c, stride=(2, 2), groups=g))
    return out


def _resnext_layers(N, size, C, g):
    """ResNeXt-50-shaped bottleneck middle layers: widths C ... 8C, stride 2 on the first layer of a stage."""
    out = []
    for i, hw in enumerate(_planes(size)[1:]):
        c = C << i
        out.append(_conv(N, c, hw, hw, c, groups=g))
        if i < 3:
            out.append(_conv(N, 2 * c, hw, hw, 2 * c, stride=(2, 2), groups=g))
    return out


def _depthwise_layers(N, size, C):
    """Depthwise layers of mobile networks: 3x3 (MobileNetV2-shaped) and 5x5, stride 1 and 2, C ... 30C channels."""
    p = _planes(size)
    table = [(3, 1, 1, p[0]), (3, 3, 2, p[0]), (3, 9, 1, p[1]), (3, 9, 2, p[1]), (3, 6, 1, p[2]), (3, 6, 2, p[2]), (3, 12, 1, p[3]),
             (3, 18, 2, p[3]), (3, 30, 1, p[4]), (5, 3, 2, p[1]), (5, 4, 1, p[2]), (5, 8, 2, p[2]), (5, 21, 1, p[3]), (5, 21, 2, p[3]),
             (5, 30, 1, p[4])]
    return [_conv(N, m * C, hw, hw, m * C, (k, k), (s, s), (k // 2, k // 2), groups=m * C) for k, m, s, hw in table]


def _pointwise_layers(N, size, C):
    """Pointwise layers around the grouped 3x3 layers of a bottleneck network (C = 64: 256 -> 128, 128 -> 256 ...)."""
    p = _planes(size)
    one, no = (1, 1), (0, 0)
    return [_conv(N, 4 * C, p[1], p[1], 2 * C, one, pad=no), _conv(N, 2 * C, p[1], p[1], 4 * C, one, pad=no),
            _conv(N, 4 * C, p[1], p[1], 8 * C, one, (2, 2), no), _conv(N, 8 * C, p[2], p[2], 4 * C, one, pad=no),
            _conv(N, 8 * C, p[3], p[3], 8 * C, one, pad=no), _conv(N, 8 * C, p[4], p[4], 8 * C, one, pad=no)]


def _general_layers(N, size, C, g):
    """Layers outside the 3x3 and pointwise families: the first layers of networks on three-channel images (3x3 and 7x7,
    stride 2), one-dimensional filters, dilated filters, 5x5 grouped filters with stride 2."""
    p = _planes(size)
    return [_conv(N, 3, size, size, C // 2, stride=(2, 2)), _conv(N, 3, size, size, C, (7, 7), (2, 2), (3, 3)),
            _conv(N, C, p[1], p[1], C, pad=(2, 2), dil=(2, 2), groups=g), _conv(N, C, p[2], p[2], C, (1, 7), pad=(0, 3), groups=g),
            _conv(N, C, p[2], p[2], C, (7, 1), pad=(3, 0), groups=g), _conv(N, C, p[2], p[2], 2 * C, (5, 5), (2, 2), (2, 2), groups=g)]


_NETWORKS = {"stack": _stack_layers, "resnet": _resnet_layers, "resnext": _resnext_layers, "general": _general_layers}
_FAMILIES = {"depthwise": _depthwise_layers, "pointwise": _pointwise_layers}


def _layers(case):
    kind, N, S, C = case["kind"], case["N"], case["size"], case["channels"]
    if kind in _NETWORKS:
        return _NETWORKS[kind](N, S, C, case["groups"])
    if kind in _FAMILIES:
        return _FAMILIES[kind](N, S, C)
    s = case.get("stride", 1)                        # one layer: "layer", "block", "host"
    return [_conv(N, C, S, case.get("width", S), case.get("channels_out", C), stride=(s, s), groups=case["groups"])]


# ---- the cases -------------------------------------------------------------------------------------------------------
def listed():
    return [
        # one small layer on one image: what a call costs (latency of a launch and of the host path)
        {"name": "one small layer", "kind": "layer", "N": 1, "size": 16, "channels": 64, "groups": 4},
        # inference on one 32x32 image through the whole grouped stack: eighteen dependent small layers
        {"name": "stack, one image", "kind": "stack", "N": 1, "size": 32, "channels": 32, "groups": 4},
        # the same stack on a batch: the workload of the benchmark's headline
        {"name": "stack, batch", "kind": "stack", "N": 128, "size": 32, "channels": 32, "groups": 8},
        # wide groups (an ordinary convolution is groups = 1) at 224x224: the tensor-core-bound end, in network order
        {"name": "resnet, groups 1", "kind": "resnet", "N": 64, "size": 224, "channels": 64, "groups": 1},
        # the same network on images and a batch nobody tuned for: planes of 50, 25, 13 and 7 pixels
        {"name": "resnet, odd sizes", "kind": "resnet", "N": 13, "size": 200, "channels": 64, "groups": 2},
        # 32 groups of 4 to 32 channels: the shape grouped convolutions are best known for
        {"name": "resnext", "kind": "resnext", "N": 64, "size": 224, "channels": 128, "groups": 32},
        # one large layer with two wide groups (the group-count sweep)
        {"name": "one large layer", "kind": "layer", "N": 32, "size": 56, "channels": 256, "groups": 2},
        # depthwise layers of mobile networks, 3x3 and 5x5, both strides
        {"name": "depthwise", "kind": "depthwise", "N": 64, "size": 224, "channels": 32},
        # the pointwise layers that re-mix channels between grouped layers
        {"name": "pointwise", "kind": "pointwise", "N": 64, "size": 224, "channels": 64},
        # the grouped 3x3 + pointwise block in one call
        {"name": "block", "kind": "block", "N": 64, "size": 56, "channels": 64, "groups": 16, "pointwise_out": 64},
        # filters of other sizes, dilation, and first layers on three-channel images
        {"name": "other filters", "kind": "general", "N": 16, "size": 224, "channels": 64, "groups": 4},
        # activations in pinned host memory: copy in, layer, copy out
        {"name": "host buffers", "kind": "host", "N": 64, "size": 56, "channels": 64, "groups": 8},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _image(rng):
    """Image sizes: half of them the usual multiples of 32, half anything."""
    return rng.choice([128, 160, 192, 224, 256]) if rng.random() < 0.5 else rng.randrange(128, 257)


def _groups_of(rng, C, most):
    return rng.choice([g for g in (1, 2, 4, 8, 16, 32, 64) if C % (2 * g) == 0 and g <= most])


def draw(rng):
    most = {}
    for c in listed():
        w = work(c)
        for key in ("bytes", "flops"):
            most[c["kind"], key] = max(most.get((c["kind"], key), 0), w[key])
    while True:
        kind = rng.choice(["layer", "layer", "stack", "resnet", "resnext", "depthwise", "pointwise", "block", "general", "host"])
        c = {"kind": kind, "N": _log_int(rng, 1, 128)}
        if kind == "layer":
            C = rng.choice([32, 48, 64, 96, 128, 192, 256])
            c.update(size=_log_int(rng, 7, 60), width=_log_int(rng, 7, 60), channels=C, channels_out=rng.choice([C, C, 2 * C]),
                     groups=_groups_of(rng, C, 64), stride=rng.choice([1, 1, 2]))
        elif kind == "stack":
            c.update(size=rng.choice([32, 32, rng.randrange(24, 41)]), channels=rng.choice([32, 48, 64]), groups=rng.choice([1, 2, 4, 8, 16]))
        elif kind == "resnet":
            C = rng.choice([32, 64, 96])
            c.update(size=_image(rng), channels=C, groups=rng.choice([1, 2, 4, 8, 16, 32]))
        elif kind == "resnext":
            c.update(size=_image(rng), channels=128, groups=rng.choice([16, 32]))
        elif kind == "depthwise":
            c.update(size=_image(rng), channels=rng.choice([16, 24, 32, 40]))
        elif kind == "pointwise":
            c.update(size=_image(rng), channels=rng.choice([32, 48, 64]))
        elif kind == "block":
            C = rng.choice([32, 64])
            c.update(size=rng.choice([8, 16, 24, 28, 32, 48, 56]), channels=C, groups=rng.choice([2, 4, 8, 16]),
                     pointwise_out=rng.choice([32, 48, 64]))
        elif kind == "general":
            c.update(N=_log_int(rng, 1, 32), size=_image(rng), channels=rng.choice([32, 64, 96]), groups=rng.choice([1, 2, 4, 8, 16]))
        else:
            C = rng.choice([32, 64, 96, 128])
            c.update(size=_log_int(rng, 7, 60), channels=C, groups=_groups_of(rng, C, 32), stride=rng.choice([1, 2]))
        w = work(c)
        if all(w[key] <= most[kind, key] for key in ("bytes", "flops")):
            return c


# ---- running a case --------------------------------------------------------------------------------------------------
class _Layer:
    """A descriptor, its packed weights and its output buffer: what a program keeps for a layer."""

    def __init__(self, L, gen, dev, stream, pointwise_out=0):
        N, Ci, H, W, Co, k, s, p, d, g = L
        self.desc = gconv.gconv_desc_create_2d(N, Ci, H, W, Co, k[0], k[1], s[0], s[1], p[0], p[1], d[0], d[1], g)
        weakref.finalize(self, gconv.gconv_desc_destroy, self.desc)
        Ho, Wo = gconv.gconv_out_shape(self.desc)
        w = torch.randn((Co, Ci // g, k[0], k[1]), generator=gen, device=dev).mul_(math.sqrt(2.0 / (Ci // g * k[0] * k[1])))
        self.c2 = pointwise_out
        if self.c2:
            w2 = torch.randn((self.c2, Co), generator=gen, device=dev).mul_(math.sqrt(2.0 / Co))
            self.wp = torch.empty(gconv.gconv_block_packed_bytes(self.desc, self.c2) // 4, device=dev)
            gconv.gconv_block_pack_weights(self.desc, self.c2, w, w2, self.wp, stream)
        else:
            self.wp = torch.empty(gconv.gconv_packed_bytes(self.desc) // 4, device=dev)
            gconv.gconv_pack_weights(self.desc, w, self.wp, stream)
            self.workspace = attach_workspace(self.desc, dev)
        self.y = torch.empty((N, self.c2 or Co, Ho, Wo), device=dev)


def prepare(case, seed):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    stream = torch.cuda.current_stream(dev)
    layers = _layers(case)

    def activations(L):
        if case["kind"] == "resnext":
            return torch.randn((L[0], L[1], L[2], L[3]), generator=gen, device=dev)
        return torch.rand((L[0], L[1], L[2], L[3]), generator=gen, device=dev).mul_(2.0).sub_(1.0)

    state = {"kind": case["kind"], "stream": stream, "layers": [_Layer(L, gen, dev, stream, case.get("pointwise_out", 0)) for L in layers]}
    if case["kind"] in ("stack", "resnet"):          # a layer reads the layer before it
        state["x"] = [activations(layers[0])] + [m.y for m in state["layers"][:-1]]
    else:
        state["x"] = [activations(L) for L in layers]
    if case["kind"] == "host":
        m = state["layers"][0]
        state["x_host"] = state["x"][0].cpu().pin_memory()
        state["y_host"] = torch.empty(m.y.shape, pin_memory=True)
    return state


def run(state):
    stream = state["stream"]
    if state["kind"] == "host":
        m = state["layers"][0]
        gconv.gconv_forward_host(m.desc, state["x_host"], m.wp, state["y_host"], state["x"][0], m.y, stream)
        return state["y_host"]
    if state["kind"] == "block":
        m = state["layers"][0]
        gconv.gconv_block_forward(m.desc, m.c2, state["x"][0], m.wp, m.y, stream)
        return m.y
    for m, x in zip(state["layers"], state["x"]):
        gconv.gconv_forward(m.desc, x, m.wp, m.y, stream)
    return [m.y for m in state["layers"]]


def work(case):
    """Each layer reads its input and its weights once and writes its output once; 2 operations a multiply-add of the
    grouped sum (the zeros of merged groups are not counted).  A fused block's intermediate is neither written nor read."""
    nbytes = flops = 0
    for L in _layers(case):
        N, Ci, H, W, Co, k, s, p, d, g = L
        Ho, Wo = _out_hw(L)
        taps = k[0] * k[1]
        C2 = case.get("pointwise_out", 0)
        nbytes += 4 * (N * Ci * H * W + N * (C2 or Co) * Ho * Wo + Co * (Ci // g) * taps + C2 * Co)
        flops += 2 * N * Co * Ho * Wo * ((Ci // g) * taps + C2)
    return {"bytes": nbytes, "flops": flops}


def _tf32(L):
    N, Ci, H, W, Co, k, s, p, d, g = L
    desc = gconv.gconv_desc_create_2d(N, Ci, H, W, Co, k[0], k[1], s[0], s[1], p[0], p[1], d[0], d[1], g)
    try:
        return gconv.gconv_variant(desc) == gconv.GCONV_VARIANT_IGEMM_TF32
    finally:
        gconv.gconv_desc_destroy(desc)


def tolerance(case):
    """About four times what the same sums in fp64 differ by: 4.2e-4 for a layer on the TF32 tensor cores (4.6e-4 with
    normal inputs) and 3.6e-4 more for every further layer of a chain, 7.7e-4 for the two contractions of a block, 3.5e-7
    for an FP32 layer."""
    layers = _layers(case)
    if not any(_tf32(L) for L in layers):
        return {"rel": 1.5e-6}
    if case["kind"] == "block":
        return {"rel": 3.1e-3}
    depth = len(layers) if case["kind"] in ("stack", "resnet") else 1
    return {"rel": 1.8e-3 + 1.45e-3 * (depth - 1)}
