"""The work that users of this library have it do, as measurable cases.

A case is one pass through the public binding (paper_1809_10572_gb300.samd):
a convolution layer, a chain of layers, or a packed operation, over the
shapes and lane formats of the repository's workloads and tests. Every output
is an integer, so every comparison is exact.
"""
import math

import torch

from paper_1809_10572_gb300 import samd

DEV = "cuda"


# ---- the cases -----------------------------------------------------------------


def listed():
    return [
        # the smallest whole call: one 16-channel 3x3 layer with its weights still
        # packed, as a program that runs a layer once calls it (latency)
        dict(name="conv_c16_call", kind="conv_call", N=1, C=16, H=32, W=32, K=16, R=3, stride=1, pad=1, ba=4, sa=0,
             bw=4, sw=1, bo=4, so=0, wb=64, acc=True, packed=True),
        # an 8-bit layer whose int32 sums are wanted (the accumulators feed float code)
        dict(name="conv_u8s8_acc", kind="conv", N=8, C=256, H=28, W=28, K=256, R=3, stride=1, pad=1, ba=8, sa=0, bw=8,
             sw=1, bo=8, so=0, wb=32, acc=True, packed=False),
        # the bit-width sweep: 32 independent 64-channel layers, b = 1..8 and all sign
        # combinations, on eight streams of one CUDA graph
        dict(name="sweep_step", kind="sweep", N=8, C=64, H=56),
        # a whole network: the 13 layers of VGG-16 at u4 x s4 with their pools, batch 16
        dict(name="vgg16_b16", kind="vgg", N=16, H=224),
        # ResNet-50 bottleneck blocks at u6 x s2, batch 64: the first (large images, few
        # channels), one that halves the image, and a late one (small images, many channels)
        dict(name="bottleneck_56", kind="bottleneck", N=64, cin=64, mid=64, cout=256, H=56, stride=1, proj=True, ba=6,
             bw=2),
        dict(name="bottleneck_28_down", kind="bottleneck", N=64, cin=512, mid=256, cout=1024, H=28, stride=2, proj=True,
             ba=6, bw=2),
        dict(name="bottleneck_7", kind="bottleneck", N=64, cin=2048, mid=512, cout=2048, H=7, stride=1, proj=False,
             ba=6, bw=2),
        # packed arithmetic on a large array
        dict(name="add_sat_u4", kind="elementwise", op="add", bits=4, signed=0, spacer=0, wb=32, n=1 << 28, sat=1,
             shift=0, bits_o=4, signed_o=0),
        # a change of format between layers: signed 8-bit lanes clamped to unsigned 4-bit ones
        dict(name="requant_s8_u4", kind="elementwise", op="requant", bits=8, signed=1, spacer=0, wb=32, n=1 << 26,
             sat=0, shift=3, bits_o=4, signed_o=0),
        # activations entering and leaving the packed form, NHWC rows of a layer's channels:
        # 64 channels are not a multiple of the 5 lanes of a 6-bit word
        dict(name="pack_u6_rows64", kind="pack", rows=64 * 56 * 56, inner=64, bits=6, signed=0, spacer=0, wb=32),
        dict(name="unpack_s4_w64", kind="unpack", rows=64 * 56 * 56, inner=256, bits=4, signed=1, spacer=0, wb=64),
        # images packed along their width, convolved by the wide-multiply engine
        dict(name="conv_nchw_u4s4", kind="conv_nchw", N=8, C=64, H=56, W=56, K=64, R=3, pad=1, ba=4, sa=0, bw=4, sw=1,
             bo=4, so=0, wb=32, acc=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _bound_ok(taps, ba, sa, bw, sw):
    a, w = _amax(ba, sa), _amax(bw, sw)
    return taps * a * w < 1 << 24 or (bw > 4 and taps * a * 16 < 1 << 24)


def _draw_conv(rng):
    while True:
        R = rng.choice([1, 3, 3, 5])
        c = dict(kind=rng.choice(["conv", "conv", "conv_call"]), N=_log(rng, 1, 64), C=_log(rng, 3, 1024),
                 H=_log(rng, 7, 224), W=0, K=_log(rng, 16, 1024), R=R, stride=rng.choice([1, 1, 1, 2]), pad=R // 2,
                 ba=rng.randint(1, 8), sa=0, bw=rng.randint(1, 8), sw=0, bo=rng.randint(1, 8),
                 so=rng.randint(0, 1), wb=rng.choice([32, 32, 32, 64]), acc=rng.random() < 0.3, packed=True)
        c["W"] = c["H"] if rng.random() < 0.7 else _log(rng, 7, 224)
        c["sa"], c["sw"] = int(c["ba"] > 1 and rng.random() < 0.4), int(c["bw"] > 1 and rng.random() < 0.7)
        if rng.random() < 0.5:  # channel counts of networks are mostly powers of two
            c["C"], c["K"] = 1 << max(4, c["C"].bit_length() - 1), 1 << max(4, c["K"].bit_length() - 1)
        if not (c["sa"] or c["sw"]) and c["bo"] == 1:
            c["so"] = 0
        if c["wb"] == 64:  # outputs in whole 64-bit words
            c["K"] = -(-c["K"] // 64) * 64
        if c["acc"] and rng.random() < 0.5:
            c["packed"] = False
        if _conv_macs(c) <= 1.5e10 and c["N"] * c["H"] * c["W"] * max(c["C"], c["K"]) <= 1 << 28 and \
                _bound_ok(R * R * c["C"], c["ba"], c["sa"], c["bw"], c["sw"]):
            return c


def draw(rng):
    kind = rng.choice(["conv", "conv", "conv", "sweep", "vgg", "bottleneck", "elementwise", "elementwise", "requant",
                       "pack", "unpack", "maxpool", "nchw"])
    if kind == "conv":
        return _draw_conv(rng)
    if kind == "sweep":
        return dict(kind="sweep", N=rng.randint(1, 8), C=rng.choice([32, 48, 64]), H=rng.choice([14, 28, 42, 56]))
    if kind == "vgg":
        return dict(kind="vgg", N=_log(rng, 1, 16), H=32 * rng.randint(2, 7))
    if kind == "bottleneck":
        mid = rng.choice([64, 128, 256, 512])
        H = 3584 // mid + rng.randint(0, 1)  # 56, 28, 14, 7, or one more
        if rng.random() < 0.5:
            return dict(kind="bottleneck", N=_log(rng, 1, 64), cin=4 * mid, mid=mid, cout=4 * mid, H=H, stride=1,
                        proj=False, ba=rng.choice([4, 6, 8]), bw=rng.choice([2, 3, 4]))
        return dict(kind="bottleneck", N=_log(rng, 1, 64), cin=2 * mid, mid=mid, cout=4 * mid, H=2 * H, stride=2,
                    proj=True, ba=rng.choice([4, 6, 8]), bw=rng.choice([2, 3, 4]))
    bits, signed, wb = rng.randint(1, 8), rng.randint(0, 1), rng.choice([32, 32, 64])
    spacer = rng.choice([0, 0, 0, 1])
    if kind in ("elementwise", "requant"):
        signed = signed if bits > 1 else 0
        op = "requant" if kind == "requant" else rng.choice(["add", "sub", "mul", "relu", "requant"])
        c = dict(kind="elementwise", op=op, bits=bits, signed=signed, spacer=spacer, wb=wb, n=_log(rng, 1 << 10, 1 << 28),
                 sat=int(op in ("add", "sub", "mul") and rng.random() < 0.5), shift=0, bits_o=bits, signed_o=signed)
        if op == "requant":
            c["shift"] = rng.randint(0, bits - 1 - signed)
        if kind == "requant":
            c["bits_o"], c["signed_o"], c["n"] = rng.randint(1, 8), rng.randint(0, 1), _log(rng, 1 << 10, 1 << 26)
        return c
    if kind in ("pack", "unpack"):
        inner = rng.choice([3, 16, 24, 32, 64, 64, 96, 128, 256, 512, _log(rng, 3, 2048)])
        return dict(kind=kind, rows=_log(rng, max(1, 4096 // inner), (1 << 25) // inner), inner=inner, bits=bits,
                    signed=signed, spacer=spacer, wb=wb)
    if kind == "maxpool":
        C = rng.choice([16, 32, 64, 96, 128, 256, 512, _log(rng, 3, 512)])
        return dict(kind="maxpool", N=_log(rng, 1, 64), C=C, H=2 * _log(rng, 2, 112), W=2 * _log(rng, 2, 112),
                    bits=bits, signed=signed, spacer=spacer, wb=wb)
    while True:
        c = dict(kind="conv_nchw", N=rng.randint(1, 8), C=_log(rng, 3, 128), H=_log(rng, 7, 64), W=_log(rng, 7, 64),
                 K=_log(rng, 16, 128), R=rng.choice([1, 3, 3]), pad=0, ba=rng.randint(1, 6), sa=0,
                 bw=rng.randint(1, 6), sw=0, bo=rng.randint(1, 8), so=rng.randint(0, 1),
                 wb=rng.choice([32, 32, 64]), acc=rng.random() < 0.5)
        c["pad"] = c["R"] // 2
        c["sa"], c["sw"] = int(c["ba"] > 1 and rng.random() < 0.4), int(c["bw"] > 1 and rng.random() < 0.7)
        if not (c["sa"] or c["sw"]) and c["bo"] == 1:
            c["so"] = 0
        bound = c["R"] * c["R"] * c["C"] * _amax(c["ba"], c["sa"]) * _amax(c["bw"], c["sw"])
        F = max(bound.bit_length() + 1, max(c["ba"], c["bw"]) + 1)
        if c["R"] * F <= 64 and bound < 1 << 31 and _conv_macs(c) <= 9e8:
            return c


# ---- shapes and work -----------------------------------------------------------


def _amax(bits, signed):
    return 1 << (bits - 1) if signed else (1 << bits) - 1


def _out(c):
    st = c.get("stride", 1)
    return (c["H"] + 2 * c["pad"] - c["R"]) // st + 1, (c["W"] + 2 * c["pad"] - c["R"]) // st + 1


def _conv_macs(c):
    ho, wo = _out(c)
    return c["N"] * ho * wo * c["K"] * c["C"] * c["R"] * c["R"]


def _layer_shift(l):
    """Requantize shift that spreads a sum of uniform products over the output lane: a sum of positive
    products lies near its mean, any other within a few deviations of zero."""
    taps, a, w = l["C"] * l["R"] * l["R"], _amax(l["ba"], l["sa"]), _amax(l["bw"], l["sw"])
    size = math.sqrt(taps) * a * w / 3 if l["sa"] or l["sw"] else taps * a * w / 4
    return max(0, math.floor(math.log2(size / 2.0 ** (l["bo"] - l["so"] - 1))))


def _conv(N, C, H, W, K, R, stride, pad, ba, sa, bw, sw, bo, so, wb, **more):
    return dict(N=N, C=C, H=H, W=W, K=K, R=R, stride=stride, pad=pad, ba=ba, sa=sa, bw=bw, sw=sw, bo=bo, so=so, wb=wb,
                **more)


def _sweep_layers(c):
    return [_conv(c["N"], c["C"], c["H"], c["H"], c["C"], 3, 1, 1, b, sa, b, sw, b, sa, 32)
            for b in range(1, 9) for sa in (0, 1) for sw in (0, 1)]


def _vgg_layers(c):
    widths = [64, 64, "P", 128, 128, "P", 256, 256, 256, "P", 512, 512, 512, "P", 512, 512, 512]
    layers, h, cin = [], c["H"], 3
    for k in widths:
        if k == "P":
            layers[-1]["pool"] = True
            h //= 2
        else:
            layers.append(_conv(c["N"], cin, h, h, k, 3, 1, 1, 4, 0, 4, 1, 4, 0, 32, pool=False))
            cin = k
    return layers


def _bottleneck_layers(c):
    N, H, st, ba, bw = c["N"], c["H"], c["stride"], c["ba"], c["bw"]
    ho = (H - 1) // st + 1
    a = _conv(N, c["cin"], H, H, c["mid"], 1, 1, 0, ba, 0, bw, 1, ba, 0, 32)
    b = _conv(N, c["mid"], H, H, c["mid"], 3, st, 1, ba, 0, bw, 1, ba, 0, 32)
    d = _conv(N, c["mid"], ho, ho, c["cout"], 1, 1, 0, ba, 0, bw, 1, ba, 0, 32)
    p = _conv(N, c["cin"], H, H, c["cout"], 1, st, 0, ba, 0, bw, 1, ba, 0, 32)
    return [a, b, d] + ([p] if c["proj"] else [])


def _layers(c):
    if c["kind"] in ("conv", "conv_call", "conv_nchw"):
        return [c]
    return {"sweep": _sweep_layers, "vgg": _vgg_layers, "bottleneck": _bottleneck_layers}[c["kind"]](c)


def _words_bytes(rows, inner, bits, spacer, wb):
    return rows * -(-inner // (wb // (bits + spacer))) * (wb // 8)


def work(c):
    kind = c["kind"]
    if kind == "elementwise":
        ins = 2 if c["op"] in ("add", "sub", "mul") else 1
        return {"bytes": ins * _words_bytes(1, c["n"], c["bits"], c["spacer"], c["wb"]) +
                _words_bytes(1, c["n"], c["bits_o"], c["spacer"], c["wb"]), "flops": 0}
    if kind in ("pack", "unpack"):
        return {"bytes": c["rows"] * c["inner"] + _words_bytes(c["rows"], c["inner"], c["bits"], c["spacer"], c["wb"]),
                "flops": 0}
    if kind == "maxpool":
        px = c["N"] * c["H"] * c["W"]
        return {"bytes": _words_bytes(px + px // 4, c["C"], c["bits"], c["spacer"], c["wb"]), "flops": 0}
    nbytes, macs = 0, 0
    for i, l in enumerate(_layers(c)):
        ho, wo = _out(dict(l))
        macs += _conv_macs(dict(l))
        if kind == "conv_nchw":
            nbytes += _words_bytes(l["N"] * l["C"] * l["H"], l["W"], l["ba"], 0, l["wb"])
            nbytes += _words_bytes(l["K"] * l["C"] * l["R"], l["R"], l["bw"], 0, l["wb"])
            nbytes += l["N"] * l["K"] * ho * wo * 4 if l["acc"] else 0
            nbytes += _words_bytes(l["N"] * l["K"] * ho, wo, l["bo"], 0, l["wb"])
            continue
        first = kind in ("conv", "conv_call", "sweep") or i == 0
        # in a chain the tensors between layers are both written and read
        nbytes += _words_bytes(l["N"] * l["H"] * l["W"], l["C"], l["ba"], 0, l["wb"]) if first else 0
        nbytes += _words_bytes(l["K"] * l["R"] * l["R"], l["C"], l["bw"], 0, l["wb"])
        nbytes += l["N"] * ho * wo * l["K"] * 4 if l.get("acc") else 0
        out = _words_bytes(l["N"] * ho * wo, l["K"], l["bo"], 0, l["wb"]) if l.get("packed", True) else 0
        nbytes += (out // 4 if l.get("pool") else out) * (1 if first and kind not in ("vgg", "bottleneck") else 2)
    return {"bytes": nbytes, "flops": 2 * macs}


def tolerance(c):
    return "exact"


# ---- inputs --------------------------------------------------------------------


def _gen(seed, k):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + 7919 * k) & 0x7FFFFFFF)


def _lanes(seed, k, shape, bits, signed):
    """Lane values uniform over the lane's range, one per byte."""
    g = _gen(seed, k)
    v = torch.randint(0, 1 << bits, shape, dtype=torch.uint8, device=DEV, generator=g)
    if signed and bits < 8:
        v = (v.view(torch.int8) << (8 - bits)) >> (8 - bits)
    return v.view(torch.int8)


def _values(lanes, signed, dtype):
    return (lanes if signed else lanes.view(torch.uint8)).to(dtype)


def _fmt(bits, signed, spacer=0, wb=32):
    return samd.fmt(bits, bool(signed), spacer, wb)


def _formats(l):
    return _fmt(l["ba"], l["sa"], 0, l["wb"]), _fmt(l["bw"], l["sw"], 0, l["wb"]), _fmt(l["bo"], l["so"], 0, l["wb"])


def _conv_shape(l):
    return samd.ConvShape(l["N"], l["C"], l["H"], l["W"], l["K"], l["R"], l["R"], l.get("stride", 1), l["pad"])


def _symmetric(seed, k, shape, bits, signed):
    """Lane values of a quantized tensor: signed ones of 2 bits and more symmetric about zero."""
    if not signed or bits == 1:
        return _lanes(seed, k, shape, bits, signed)
    top = (1 << (bits - 1)) - 1
    return torch.randint(-top, top + 1, shape, dtype=torch.int8, device=DEV, generator=_gen(seed, k))


def _act_lanes(l, seed, i):
    return _symmetric(seed, 2 * i, (l["N"], l["H"], l["W"], l["C"]), l["ba"], l["sa"])


def _wt_lanes(l, seed, i):
    return _symmetric(seed, 2 * i + 1, (l["K"], l["R"], l["R"], l["C"]), l["bw"], l["sw"])


def _pack_act(l, seed, i):
    return samd.pack(_act_lanes(l, seed, i), _formats(l)[0])


def _prepared(l, seed, i, packed=True):
    fa, fw, fo = _formats(l)
    w = samd.pack(_wt_lanes(l, seed, i), fw)
    return samd.PreparedConv(w, _conv_shape(l), fa, fw, fo if packed else None)


def _captured(once):
    """once()'s launches in a CUDA graph, as a program that repeats a fixed step keeps it."""
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        once(stream)
    torch.cuda.current_stream().wait_stream(stream)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        once(stream)
    return graph


def _prepare_sweep(c, seed):
    layers = _sweep_layers(c)
    acts = [_pack_act(l, seed, i) for i, l in enumerate(layers)]
    convs = [_prepared(l, seed, i) for i, l in enumerate(layers)]
    outs = [p.outputs(want_acc=False)[1] for p in convs]
    shifts = [_layer_shift(l) for l in layers]
    side = [torch.cuda.Stream() for _ in range(8)]

    def once(stream):
        for s in side:
            s.wait_stream(stream)
        for i, p in enumerate(convs):
            p(acts[i], None, outs[i], shift=shifts[i], stream=side[i % 8])
        for s in side:
            stream.wait_stream(s)

    samd.samd_conv2d_set_min_tiles_per_cta(8)  # many layers at once: fewer SMs for each
    try:
        graph = _captured(once)
    finally:
        samd.samd_conv2d_set_min_tiles_per_cta(4)
    return dict(graph=graph, outs=outs, keep=(acts, convs, side))


def _prepare_vgg(c, seed):
    layers = _vgg_layers(c)
    x = _pack_act(layers[0], seed, 0)
    convs = [_prepared(l, seed, i) for i, l in enumerate(layers)]
    steps, outs = [], []
    for l, p in zip(layers, convs):
        fused = l["pool"] and p.pool2x2_supported()
        f = _formats(l)[2]
        full = None if fused else p.outputs(want_acc=False)[1]
        pooled = samd.empty_words(f, l["N"] * (l["H"] // 2) * (l["W"] // 2), l["K"]) if l["pool"] else None
        steps.append((l, p, f, _layer_shift(l), full, pooled))
        outs.append(pooled if l["pool"] else full)

    def once(stream):
        t = x
        for l, p, f, shift, full, pooled in steps:
            if full is None:
                t = p.pool2x2(t, pooled, shift=shift, stream=stream)
                continue
            p(t, None, full, shift=shift, stream=stream)
            t = full
            if pooled is not None:
                samd.samd_maxpool2x2(f, full, pooled, l["N"], l["K"], l["H"], l["W"], stream=stream)
                t = pooled

    return dict(graph=_captured(once), outs=outs, keep=(x, convs, steps))


def prepare(c, seed):
    kind = c["kind"]
    if kind == "sweep":
        return dict(_prepare_sweep(c, seed), kind=kind)
    if kind == "vgg":
        return dict(_prepare_vgg(c, seed), kind=kind)
    if kind == "bottleneck":
        layers = _bottleneck_layers(c)
        convs = [_prepared(l, seed, i) for i, l in enumerate(layers)]
        f = _formats(layers[0])[0]
        return dict(kind=kind, x=_pack_act(layers[0], seed, 0), convs=convs, f=f,
                    outs=[p.outputs(want_acc=False)[1] for p in convs], shifts=[_layer_shift(l) for l in layers],
                    y=samd.empty_words(f, layers[2]["N"] * _out(layers[2])[0] * _out(layers[2])[1], c["cout"]))
    if kind == "conv":
        p = _prepared(c, seed, 0, c["packed"])
        acc, packed = p.outputs(c["acc"], c["packed"])
        return dict(kind=kind, conv=p, x=_pack_act(c, seed, 0), acc=acc, packed=packed, shift=_layer_shift(c))
    if kind == "conv_call":
        fa, fw, fo = _formats(c)
        return dict(kind=kind, shape=_conv_shape(c), fa=fa, fw=fw, fo=fo if c["packed"] else None, acc=c["acc"],
                    x=_pack_act(c, seed, 0), w=samd.pack(_wt_lanes(c, seed, 0), fw), shift=_layer_shift(c))
    if kind == "conv_nchw":
        fa, fw, fo = _formats(c)
        x, w = _act_lanes(c, seed, 0).permute(0, 3, 1, 2), _wt_lanes(c, seed, 0).permute(0, 3, 1, 2)
        return dict(kind=kind, shape=_conv_shape(c), fa=fa, fw=fw, fo=fo, acc=c["acc"], x=samd.pack(x, fa),
                    w=samd.pack(w, fw), shift=_layer_shift(c))
    if kind == "elementwise":
        fa, fo = _fmt(c["bits"], c["signed"], c["spacer"], c["wb"]), _fmt(c["bits_o"], c["signed_o"], c["spacer"], c["wb"])
        a = samd.pack(_lanes(seed, 0, (c["n"],), c["bits"], c["signed"]), fa)
        two = c["op"] in ("add", "sub", "mul")
        b = samd.pack(_lanes(seed, 1, (c["n"],), c["bits"], c["signed"]), fa) if two else None
        return dict(kind=kind, op=c["op"], a=a, b=b, fa=fa, fo=fo, n=c["n"], shift=c["shift"], sat=bool(c["sat"]),
                    out=samd.empty_words(fo, 1, c["n"]))
    f = _fmt(c["bits"], c["signed"], c["spacer"], c["wb"])
    if kind == "maxpool":
        x = samd.pack(_lanes(seed, 0, (c["N"], c["H"], c["W"], c["C"]), c["bits"], c["signed"]), f)
        out = samd.empty_words(f, c["N"] * (c["H"] // 2) * (c["W"] // 2), c["C"])
        return dict(kind=kind, f=f, x=x, out=out, dims=(c["N"], c["C"], c["H"], c["W"]))
    x = _lanes(seed, 0, (c["rows"], c["inner"]), c["bits"], c["signed"])
    if kind == "pack":
        return dict(kind=kind, f=f, x=x, rows=c["rows"], inner=c["inner"], out=samd.empty_words(f, c["rows"], c["inner"]))
    return dict(kind=kind, f=f, x=samd.pack(x, f), rows=c["rows"], inner=c["inner"],
                out=torch.empty(c["rows"], c["inner"], dtype=torch.int8, device=DEV))


# ---- one pass ------------------------------------------------------------------


def run(s):
    kind = s["kind"]
    if kind in ("sweep", "vgg"):
        s["graph"].replay()
        return s["outs"]
    if kind == "bottleneck":
        (a, b, d), o, sh = s["convs"][:3], s["outs"], s["shifts"]
        a(s["x"], None, o[0], shift=sh[0])
        b(o[0], None, o[1], shift=sh[1])
        d(o[1], None, o[2], shift=sh[2])
        skip = s["x"]
        if len(o) > 3:
            s["convs"][3](s["x"], None, o[3], shift=sh[3])
            skip = o[3]
        y = s["y"]  # the residual sum, clamped to the lane; whole words, so their padding lanes stay zero
        samd.samd_elementwise("add", s["f"], o[2], skip, s["f"], y, y.numel() * samd.samd_lanes_per_word(s["f"]), 0, 1)
        return o + [y]
    if kind == "conv":
        s["conv"](s["x"], s["acc"], s["packed"], shift=s["shift"])
        return [t for t in (s["acc"], s["packed"]) if t is not None]
    if kind in ("conv_call", "conv_nchw"):
        f = samd.conv2d if kind == "conv_call" else samd.conv2d_nchw
        acc, packed = f(s["x"], s["w"], s["shape"], s["fa"], s["fw"], s["fo"], shift=s["shift"], want_acc=s["acc"])
        return [t for t in (acc, packed) if t is not None]
    if kind == "elementwise":
        return samd.elementwise(s["op"], s["a"], s["b"], s["fa"], s["n"], fo=s["fo"], shift=s["shift"],
                                saturate=s["sat"], out=s["out"])
    if kind == "maxpool":
        N, C, H, W = s["dims"]
        samd.samd_maxpool2x2(s["f"], s["x"], s["out"], N, C, H, W)
    elif kind == "pack":
        samd.samd_pack(s["f"], s["x"], s["out"], s["rows"], s["inner"])
    else:
        samd.samd_unpack(s["f"], s["x"], s["out"], s["rows"], s["inner"])
    return s["out"]


# ---- the same in plain torch -----------------------------------------------------


def _words(v, bits, spacer, wb):
    """Rows (last axis) of integer lanes -> flat words, least significant lane first."""
    inner = v.shape[-1]
    v = v.reshape(-1, inner)
    L = wb // (bits + spacer)
    wpr = -(-inner // L)
    w = torch.zeros((v.shape[0], wpr), dtype=torch.int64, device=v.device)
    for i in range(L):
        lane = v[:, i::L].to(torch.int64) & ((1 << bits) - 1)
        w[:, :lane.shape[1]] |= lane << (i * (bits + spacer))
    return w.reshape(-1).to(torch.int32 if wb == 32 else torch.int64)


def _clamp(v, bits, signed):
    return v.clamp(-(1 << (bits - 1)) if signed else 0, (1 << (bits - 1)) - 1 if signed else (1 << bits) - 1)


def _exact_conv(x, w, l):
    """x: N H W C, w: K R S C, both float64 integers -> int64 N Ho Wo K."""
    ho, wo = _out(dict(l))
    st, p = l.get("stride", 1), l["pad"]
    x = torch.nn.functional.pad(x, (0, 0, p, p, p, p))
    acc = torch.zeros((l["N"] * ho * wo, l["K"]), dtype=torch.float64, device=x.device)
    for r in range(l["R"]):
        for s in range(l["R"]):
            t = x[:, r:r + (ho - 1) * st + 1:st, s:s + (wo - 1) * st + 1:st].reshape(-1, l["C"])
            acc.addmm_(t, w[:, r, s].t())
    return acc.to(torch.int64).reshape(l["N"], ho, wo, l["K"])


def _requant(acc, l):
    return _clamp(acc >> _layer_shift(l), l["bo"], l["so"])


def _pool(v):
    return torch.maximum(torch.maximum(v[:, ::2, ::2], v[:, 1::2, ::2]), torch.maximum(v[:, ::2, 1::2], v[:, 1::2, 1::2]))


def exact(c, seed):
    kind = c["kind"]
    d = torch.float64
    if kind in ("conv", "conv_call", "conv_nchw"):
        acc = _exact_conv(_values(_act_lanes(c, seed, 0), c["sa"], d), _values(_wt_lanes(c, seed, 0), c["sw"], d), c)
        if kind == "conv_nchw":
            acc = acc.permute(0, 3, 1, 2).contiguous()
        out = [acc.to(torch.int32)] if c["acc"] else []
        return out + ([_words(_requant(acc, c), c["bo"], 0, c["wb"])] if c.get("packed", True) else [])
    if kind in ("sweep", "vgg", "bottleneck"):
        layers = _layers(c)
        x = _values(_act_lanes(layers[0], seed, 0), layers[0]["sa"], d)
        first, outs, y = x, [], None
        for i, l in enumerate(layers):
            if kind == "sweep":
                x = _values(_act_lanes(l, seed, i), l["sa"], d)
            elif kind == "bottleneck" and i == 3:
                main, x = y, first
            y = _requant(_exact_conv(x, _values(_wt_lanes(l, seed, i), l["sw"], d), l), l)
            if l.get("pool"):
                y = _pool(y)
            outs.append(_words(y, l["bo"], 0, l["wb"]))
            x = y.to(d)
        if kind == "bottleneck":
            main, skip = (main, y) if c["proj"] else (y, first.to(torch.int64))
            outs.append(_words(_clamp(main + skip, c["ba"], 0), c["ba"], 0, 32))
        return outs
    if kind == "elementwise":
        two = c["op"] in ("add", "sub", "mul")
        a = _values(_lanes(seed, 0, (c["n"],), c["bits"], c["signed"]), c["signed"], torch.int32)
        b = _values(_lanes(seed, 1, (c["n"],), c["bits"], c["signed"]), c["signed"], torch.int32) if two else None
        v = {"add": lambda: a + b, "sub": lambda: a - b, "mul": lambda: a * b, "relu": lambda: a.clamp(min=0),
             "requant": lambda: a >> c["shift"]}[c["op"]]()
        if c["sat"] or c["op"] == "requant":
            v = _clamp(v, c["bits_o"], c["signed_o"])
        return _words(v, c["bits_o"], c["spacer"], c["wb"])
    if kind == "maxpool":
        v = _values(_lanes(seed, 0, (c["N"], c["H"], c["W"], c["C"]), c["bits"], c["signed"]), c["signed"], torch.int32)
        return _words(_pool(v), c["bits"], c["spacer"], c["wb"])
    x = _lanes(seed, 0, (c["rows"], c["inner"]), c["bits"], c["signed"])
    return x if kind == "unpack" else _words(_values(x, c["signed"], torch.int32), c["bits"], c["spacer"], c["wb"])
