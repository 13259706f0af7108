"""Timed cases of the library: what a user's program has it compute, through its public entry points.

Each case is one of these uses (the "use" of a case):

  layer      one quantized convolution, filters prepared once (PreparedConv: a served model's layer) or handed over
             with the call (conv_hwc: filters that still change, a layer used once), at INT-8, INT-4 or INT-2
  staircase  the threshold compression of INT-4 / INT-2 layers (conv_hwc_thresholds)
  binary     the INT-1 convolution (conv_binary)
  net        the CIFAR-10-shaped network: three convolutions with fused 2x2 max-pooling and the fully connected layer
  block      a sub-byte layer between INT-8 neighbours: pack, convolution, 2x2 max-pool, unpack

Every output is a whole number, so results are compared bit for bit.
"""
from __future__ import annotations

import math

import torch

from paper_1908_11263_gb300 import qnn

DEV = "cuda"


def _conv(name, n, h, w, c, m, kh, kw, **more):
    case = dict(use="layer", n=n, h=h, w=w, c=c, m=m, kh=kh, kw=kw, stride=1, pad=kh // 2, bits=8, prepared=True,
                per_channel_shift=False)
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # One image through the 16x16x32 -> 64 benchmark layer: a single inference, where latency is all.
        _conv("layer_n1", 1, 16, 16, 32, 64, 3, 3),
        # The benchmark layer at its usual batch: a served INT-8 layer.
        _conv("layer_n512", 512, 16, 16, 32, 64, 3, 3),
        # The same layer at INT-4 with thresholds per channel, the compression of batch-normalised sub-byte layers.
        _conv("staircase_int4_n512", 512, 16, 16, 32, 64, 3, 3, use="staircase", bits=4, prepared=False),
        # An INT-2 layer whose neighbours work on INT-8: pack its input, convolve, pool, unpack the result.
        _conv("block_int2_n2048", 2048, 16, 16, 32, 64, 3, 3, use="block", bits=2, prepared=False),
        # Binary network layer (INT-1), the same sizes.
        _conv("binary_n512", 512, 16, 16, 32, 64, 3, 3, use="binary", bits=1, prepared=False),
        # The whole CIFAR-10-shaped network at batch 1024.
        dict(name="cifar_n1024", use="net", n=1024),
        # Layers of the ImageNet-sized networks, prepared, with a shift per channel: many pixels and few channels ...
        _conv("conv3x3_56_n256", 256, 56, 56, 64, 64, 3, 3, per_channel_shift=True),
        # ... then fewer pixels and more channels ...
        _conv("conv3x3_28_n64", 64, 28, 28, 128, 128, 3, 3, per_channel_shift=True),
        _conv("conv3x3_14_n64", 64, 14, 14, 256, 256, 3, 3, per_channel_shift=True),
        # ... and the 1x1 layers between them.
        _conv("conv1x1_14_n64", 64, 14, 14, 256, 512, 1, 1, per_channel_shift=True),
        # The stride-2 layer that halves the image between two stages of such a network.
        _conv("downsample_56_n64", 64, 56, 56, 64, 128, 3, 3, stride=2, prepared=False),
        # A layer with odd sizes throughout: image rows and filters that fill no vector, tile or block.
        _conv("ragged_n37", 37, 33, 45, 20, 44, 3, 3, prepared=False),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], uniform over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# multiply-accumulates of the largest listed layer of each kind bound the drawn ones
_MOST = 256 * 56 * 56 * 64 * 64 * 9
_MOST_STRIDED = 64 * 28 * 28 * 64 * 128 * 9


def _most_images(most, macs_per_image, limit):
    return max(1, min(limit, most // max(1, macs_per_image)))


def draw(rng):
    kind = rng.choice(["layer", "layer", "wide", "wide", "strided", "ragged", "staircase", "block", "binary", "net"])
    if kind == "net":
        return dict(use="net", n=_log(rng, 1, 2048))
    if kind == "wide":  # layers of the ImageNet-sized networks, any channel count in steps of 16
        size = rng.choice([7, 14, 28, 56, rng.randint(7, 56)])
        c, m, k = 16 * rng.randint(4, 16), 16 * rng.randint(4, 32), rng.choice([1, 3])
        case = _conv("", 1, size, size, c, m, k, k, per_channel_shift=rng.random() < 0.5)
        case["n"] = _log(rng, 1, _most_images(_MOST // 4, size * size * c * m * k * k, 128))
        return case
    if kind == "strided":  # stride 2, or 2 x 1 as for signals and spectrograms
        c, m, k = rng.choice([3, 16, 32, 4 * rng.randint(2, 32)]), 8 * rng.randint(2, 32), rng.choice([1, 3, 3, 5])
        case = _conv("", 1, rng.randint(12, 64), rng.randint(12, 64), c, m, k, k, stride=2, prepared=False,
                     per_channel_shift=rng.random() < 0.3)
        case["n"] = _log(rng, 1, _most_images(_MOST_STRIDED, case["h"] * case["w"] // 4 * c * m * k * k, 128))
        return case
    if kind == "ragged":  # odd widths and channel counts
        c, m = rng.randint(3, 60), rng.randint(5, 96)
        k = rng.choice([1, 3, 3, 5])
        case = _conv("", 1, rng.randint(9, 61), 2 * rng.randint(4, 30) + 1, c, m, k, rng.choice([k, 3]), prepared=False)
        case["n"] = _log(rng, 1, _most_images(_MOST_STRIDED // 4, case["h"] * case["w"] * c * m * k * case["kw"], 64))
        return case
    # the benchmark layer's family
    c, m, k = 32 * rng.randint(1, 2), 8 * rng.randint(2, 16), rng.choice([1, 3, 3, 5])
    case = _conv("", 1, rng.randint(7, 34), 4 * rng.randint(2, 8), c, m, k, k)
    if kind == "layer":
        case.update(bits=rng.choice([8, 8, 4, 2]), prepared=rng.random() < 0.6, per_channel_shift=rng.random() < 0.3)
    elif kind == "staircase":
        case.update(use="staircase", bits=rng.choice([4, 2]), prepared=False)
    elif kind == "block":
        case.update(use="block", bits=rng.choice([4, 2]), prepared=False)
    else:
        case.update(use="binary", bits=1, prepared=False, stride=rng.choice([1, 1, 1, 2]))
    case["n"] = _log(rng, 1, _most_images(_MOST // 4, case["h"] * case["w"] * c * m * k * k, 2048))
    return case


# the CIFAR-10-shaped network: (h, w, c, m, k) of its convolutions, each followed by a 2x2 max-pool, and its last layer
NET = [(32, 32, 3, 32, 5), (16, 16, 32, 32, 5), (8, 8, 32, 64, 5)]
NET_FC = (1024, 10)


def _out(case):
    oh = (case["h"] + 2 * case["pad"] - case["kh"]) // case["stride"] + 1
    ow = (case["w"] + 2 * case["pad"] - case["kw"]) // case["stride"] + 1
    return oh, ow


def _macs(case):
    if case["use"] == "net":
        return case["n"] * (sum(h * w * c * m * k * k for h, w, c, m, k in NET) + NET_FC[0] * NET_FC[1])
    oh, ow = _out(case)
    return case["n"] * oh * ow * case["m"] * case["kh"] * case["kw"] * case["c"]


def work(case):
    """Multiply-accumulates count twice; bytes are the inputs, filters and constants in and the results out."""
    n = case["n"]
    if case["use"] == "net":
        inner = sum((h // 2) * (w // 2) * m for h, w, _, m, _ in NET)
        filters = sum(c * m * k * k + 10 * m for _, _, c, m, k in NET) + NET_FC[0] * NET_FC[1] + 4 * NET_FC[1]
        return {"bytes": n * (32 * 32 * 3 + inner + 4 * NET_FC[1]) + filters, "flops": 2 * _macs(case)}
    oh, ow = _out(case)
    x, y, q = n * case["h"] * case["w"] * case["c"], n * oh * ow * case["m"], case["bits"]
    consts = case["m"] * (4 * ((1 << q) - 1) if case["use"] in ("staircase", "binary") else 10 + case["per_channel_shift"])
    filters = case["m"] * case["kh"] * case["kw"] * case["c"] * q // 8 + consts
    if case["use"] == "block":  # INT-8 in, pooled INT-8 out
        return {"bytes": x + n * (oh // 2) * (ow // 2) * case["m"] + filters, "flops": 2 * _macs(case)}
    return {"bytes": (x + y) * q // 8 + filters, "flops": 2 * _macs(case)}


# ---------------------------------------------------------------- inputs


class _Draw:
    """Whole numbers on the GPU from one seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed))

    def ints(self, lo, hi, shape, dtype=torch.int32):
        """Uniform in [lo, hi]."""
        return torch.randint(lo, hi + 1, shape, generator=self.g, device=DEV, dtype=torch.int64).to(dtype) \
            if math.prod(shape) < 1 << 20 else \
            torch.randint(lo, hi + 1, shape, generator=self.g, device=DEV, dtype=torch.int16).to(dtype)


def _spread(taps, bits):
    """Mean and standard deviation of an accumulator over uniform activations and weights."""
    if bits == 1:  # matching bits
        return taps / 2, math.sqrt(taps) / 2
    top, half = (1 << bits) - 1, 1 << (bits - 1)
    xx, ww = top * (2 * top + 1) / 6, (2 * half * half + 1) / 6
    return -0.5 * taps * top / 2, math.sqrt(taps * (xx * ww - (top / 4) ** 2))


def _values(case, seed):
    """The layer's integers, unpacked."""
    d = _Draw(seed)
    q, m, c = case["bits"], case["m"], case["c"]
    lo, hi = (0, 1) if q == 1 else (-(1 << (q - 1)), (1 << (q - 1)) - 1)
    v = {"x": d.ints(0, (1 << q) - 1, (case["n"], case["h"], case["w"], c), torch.uint8),
         "w": d.ints(lo, hi, (m, case["kh"], case["kw"], c), torch.int8)}
    mean, std = _spread(case["kh"] * case["kw"] * c, q)
    if case["use"] in ("staircase", "binary"):
        # thresholds at the accumulator's quantiles, shifted per channel, ascending
        steps = (1 << q) - 1
        p = (torch.arange(1, steps + 1, device=DEV, dtype=torch.float64)) / (steps + 1)
        at = mean + std * (math.sqrt(2) * torch.erfinv(2 * p - 1) +
                           d.ints(-1000, 1000, (m, 1)).double() / 1000 + d.ints(-100, 100, (m, steps)).double() / 1000)
        v["thr"] = at.round().to(torch.int32).sort(dim=1).values.contiguous()
        return v
    # batch-normalisation constants: bias within a standard deviation, kappa and lambda as fixed-point scale and offset,
    # the shift that leaves a few per cent of the outputs at the upper clip
    b = max(1, int(std))
    v["bias"] = d.ints(-b, b, (m,)) - int(mean)
    v["kappa"] = d.ints(1, 64, (m,), torch.int16)
    v["lam"] = d.ints(-(1 << 15), 1 << 15, (m,)) if q == 8 else d.ints(-16, 16, (m,))
    v["shift"] = max(0, math.ceil(math.log2(1.6 * std * 32.5 / ((1 << q) - 1))))
    if case["per_channel_shift"]:
        v["shifts"] = (v["shift"] + d.ints(-1, 1, (m,))).clamp(0, 62).to(torch.uint8)
    return v


def _pack(t, bits):
    """Q-bit values along the last dimension as packed bytes, the first element in the low bits."""
    per = 8 // bits
    if per == 1:
        return t
    f = (t.to(torch.uint8) & ((1 << bits) - 1)).view(*t.shape[:-1], t.shape[-1] // per, per)
    out = torch.zeros(f.shape[:-1], dtype=torch.uint8, device=t.device)
    for k in range(per):
        out |= f[..., k] << (k * bits)
    return out


def _net_case(case, i):
    h, w, c, m, k = NET[i]
    return dict(use="layer", n=case["n"], h=h, w=w, c=c, m=m, kh=k, kw=k, stride=1, pad=k // 2, bits=8,
                per_channel_shift=False)


def _net_values(case, seed):
    layers = [_values(dict(_net_case(case, i), n=case["n"] if i == 0 else 1), 16 * seed + i) for i in range(3)]
    d = _Draw(16 * seed + 7)
    k, m = NET_FC
    return layers, d.ints(-128, 127, (m, k), torch.int8), d.ints(-4096, 4096, (m,))


def prepare(case, seed):
    if case["use"] == "net":
        layers, fw, fb = _net_values(case, seed)
        n = case["n"]
        s = {"use": "net", "x": layers[0]["x"].contiguous(), "fw": fw, "fb": fb, "n": n, "convs": [], "outs": []}
        for (h, w, c, m, k), v in zip(NET, layers):
            s["convs"].append(qnn.PreparedConv(v["w"], v["kappa"], v["lam"], n=n, h=h, wd=w, bias=v["bias"],
                                               shift=v["shift"], bits=8, stride=1, pad=k // 2))
            s["outs"].append(torch.empty((n, h // 2, w // 2, m), dtype=torch.uint8, device=DEV))
        return s
    v = _values(case, seed)
    q = case["bits"]
    s = {"use": case["use"], "case": case, "shift": v.get("shift"), "bias": v.get("bias"), "kappa": v.get("kappa"),
         "lam": v.get("lam"), "shifts": v.get("shifts"), "thr": v.get("thr")}
    w = v["w"]
    # (the filters of an INT-8 layer are int8 tensors, packed ones uint8)
    s["w"] = w if q == 8 else _pack(w, q).contiguous()
    if case["use"] == "block":
        s["x"] = v["x"].to(torch.int8)  # the INT-8 neighbour's tensor, its values in the Q-bit range
    else:
        s["x"] = _pack(v["x"], q).contiguous()
    if case["use"] == "binary":
        s["thr"] = s["thr"].view(-1).contiguous()
    # (layers on the CUDA-core kernel have nothing to prepare)
    desc = qnn.conv_desc(case["n"], case["h"], case["w"], case["c"], case["m"], case["kh"], case["kw"], case["stride"],
                         _pads(case), q, 0) if q > 1 else None
    if case["use"] == "layer" and case["prepared"] and qnn.conv_algo(desc) == qnn.ALGO_TENSORCORE:
        s["conv"] = qnn.PreparedConv(s["w"], s["kappa"], s["lam"], n=case["n"], h=case["h"], wd=case["w"],
                                     bias=s["bias"], shifts=s["shifts"], shift=s["shift"], bits=q,
                                     stride=case["stride"], pad=_pads(case))
        s["out"] = torch.empty(s["conv"].out_shape, dtype=torch.uint8, device=DEV)
    return s


def _pads(case):
    return (case["pad"], case["pad"])


def run(s):
    if s["use"] == "net":
        x, maps = s["x"], []
        for conv, out in zip(s["convs"], s["outs"]):
            x = conv.pool2(x, out=out)
            maps.append(x)
        return {"maps": maps, "logits": qnn.linear(x.view(s["n"], -1), s["fw"], s["fb"])}
    case = s["case"]
    if "conv" in s:
        return s["conv"](s["x"], out=s["out"])
    if s["use"] == "staircase":
        return qnn.conv_hwc_thresholds(s["x"], s["w"], s["thr"], bits=case["bits"], stride=case["stride"],
                                       pad=_pads(case))
    if s["use"] == "binary":
        return qnn.conv_binary(s["x"], s["w"], s["thr"], stride=case["stride"], pad=_pads(case))
    if s["use"] == "block":
        q = case["bits"]
        x = qnn.pack_subbyte(s["x"], q)
        y = qnn.conv_hwc(x, s["w"], s["kappa"], s["lam"], bias=s["bias"], shifts=s["shifts"], shift=s["shift"], bits=q,
                         stride=case["stride"], pad=_pads(case))
        y = qnn.maxpool(y, 2, 2, q)
        return qnn.unpack_subbyte(y, q, False)
    return qnn.conv_hwc(s["x"], s["w"], s["kappa"], s["lam"], bias=s["bias"], shifts=s["shifts"], shift=s["shift"],
                        bits=case["bits"], stride=case["stride"], pad=_pads(case))


# ---------------------------------------------------------------- the same in 64 bits


def _acc(x, w, stride, pad):
    """Accumulators [n, oh, ow, m] (float64, exact for these magnitudes) of NHWC x and [m][kh][kw][c] w."""
    n, h, wd, _ = x.shape
    m, kh, kw, _ = w.shape
    xp = torch.nn.functional.pad(x.double(), (0, 0, pad, pad, pad, pad))
    oh, ow = (h + 2 * pad - kh) // stride + 1, (wd + 2 * pad - kw) // stride + 1
    out = torch.zeros((n, oh, ow, m), dtype=torch.float64, device=x.device)
    for i in range(kh):
        for j in range(kw):
            out += xp[:, i:i + stride * (oh - 1) + 1:stride, j:j + stride * (ow - 1) + 1:stride] @ w[:, i, j].double().T
    return out


def _scale_clip(acc, v, bits):
    t = (acc.to(torch.int64) + v["bias"].to(torch.int64)) * v["kappa"].to(torch.int64) + v["lam"].to(torch.int64)
    t >>= v["shifts"].to(torch.int64) if v.get("shifts") is not None else v["shift"]
    return t.clamp(0, (1 << bits) - 1).to(torch.uint8)


def _pool(y):
    n, h, w, m = y.shape
    return y[:, :h // 2 * 2, :w // 2 * 2].reshape(n, h // 2, 2, w // 2, 2, m).amax(dim=(2, 4))


def exact(case, seed):
    if _macs(case) > 4 << 30:
        return None  # double precision runs these layers too slowly
    if case["use"] == "net":
        layers, fw, fb = _net_values(case, seed)
        x, maps = layers[0]["x"], []
        for (_, _, _, _, k), v in zip(NET, layers):
            x = _pool(_scale_clip(_acc(x, v["w"], 1, k // 2), v, 8))
            maps.append(x)
        logits = x.reshape(case["n"], -1).double() @ fw.double().T + fb.double()
        return {"maps": maps, "logits": logits.to(torch.int32)}
    v = _values(case, seed)
    q = case["bits"]
    if case["use"] == "binary":
        # matching bits inside the image: (sum of products of +1 / -1 values + positions inside the image) / 2
        x, w = 2 * v["x"].to(torch.int16) - 1, 2 * v["w"].to(torch.int16) - 1
        inside = _acc(torch.ones_like(x[:1]), torch.ones_like(w[:1]), case["stride"], case["pad"])
        acc = (_acc(x, w, case["stride"], case["pad"]) + inside) / 2
        return _pack((acc >= v["thr"].view(-1).double()).to(torch.uint8), 1)
    acc = _acc(v["x"], v["w"], case["stride"], case["pad"])
    if case["use"] == "staircase":
        y = torch.zeros(acc.shape, dtype=torch.uint8, device=acc.device)
        for k in range((1 << q) - 1):
            y += (acc >= v["thr"][:, k].double()).to(torch.uint8)
        return _pack(y, q)
    y = _scale_clip(acc, v, q)
    if case["use"] == "block":
        return _pool(y).to(torch.int8)
    return _pack(y, q)
