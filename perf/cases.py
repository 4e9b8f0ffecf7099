"""What the library's speed is judged by: passes of the work that a forward-only FP16 program has
it do, through the public entry points, as eager calls on the current stream.

Kinds of case
  layer    one convolution layer of any shape (NCHW or channels-last)
  net      every convolution layer of a network in order.  A layer reads its predecessor's output
           where the shapes fit, and an input of its own where the program puts another operation
           (pooling) in between
  blocks   MobileNet as a stem and depthwise + pointwise block kernels, channels-last
  host     `net` from and to pinned host memory (hgc_conv_forward_host)
  fc       a classifier's inner-product layers
  bn       batch norm with statistics taken from the batch, or with stored ones
  load     a model's preparation: FP32 weights cast, batch norms folded in, weights registered
"""
import math

import torch

from paper_1901_00858_b200 import binding as hgc
from paper_1901_00858_b200 import workloads

NETS = {"alexnet_pair": 1, "vgg16": 2, "mobilenet_v1": 3, "resnet50": 4}
CHANNELS_LAST = hgc.HGC_FLAG_X_NHWC | hgc.HGC_FLAG_Y_NHWC


def _layer(n, c, h, w, k, r, s, pad_h, pad_w, stride, dil=1, group=1, nhwc=False, bias=True, relu=True):
    return dict(kind="layer", n=n, c=c, h=h, w=w, k=k, r=r, s=s, pad_h=pad_h, pad_w=pad_w, stride=stride, dil=dil,
                group=group, nhwc=nhwc, bias=bias, relu=relu)


def listed():
    return [
        # the smallest call: one 3x3 layer of one 32x32 image; what a call costs at all
        dict(name="single3x3_n1", **_layer(1, 3, 32, 32, 16, 3, 3, 1, 1, 1)),
        # a layer of no round size: odd channels, an odd, wide plane, a few images
        dict(name="odd_layer_n6", **_layer(6, 99, 53, 67, 161, 3, 3, 1, 1, 1)),
        # one image through 13 layers: the latency of an interactive program
        dict(name="vgg16_n1", kind="net", net="vgg16", n=1, side=224, nhwc=False),
        # the headline: 13 large 3x3 layers at batch 16, tensor bound
        dict(name="vgg16_n16", kind="net", net="vgg16", n=16, side=224, nhwc=False),
        # depthwise and pointwise layers, HBM bound, one after the other
        dict(name="mobilenet_v1_n32", kind="net", net="mobilenet_v1", n=32, side=224, nhwc=False),
        # throughput serving: 49 layers at batch 64, 1x1 layers and strided ones among them
        dict(name="resnet50_n64", kind="net", net="resnet50", n=64, side=224, nhwc=False),
        # the same layers with activations kept channels-last in between, an ordinary batch
        dict(name="resnet50_nhwc_n16", kind="net", net="resnet50", n=16, side=224, nhwc=True),
        # MobileNet's blocks as one kernel each
        dict(name="mobilenet_blocks_n8", kind="blocks", n=8, side=224),
        # requests that arrive in host memory and are answered there
        dict(name="vgg16_host_n4", kind="host", net="vgg16", n=4, side=224),
        # a classifier's three inner products: weights streamed once for few images
        dict(name="classifier_n64", kind="fc", n=64, c=25088, hidden=4096, k=1000),
        # batch norm of a first-block activation, statistics computed
        dict(name="batchnorm_n16", kind="bn", n=16, c=64, h=224, w=224, stored=False),
        # start-up of a program: 49 layers' weights from FP32 blobs
        dict(name="load_resnet50", kind="load", net="resnet50"),
    ]


# ---- shapes -------------------------------------------------------------------------------------

def _conv(n, c, h, w, k, r, s, pad_h, pad_w, stride, dil, group, nhwc, bias, relu):
    p = (h + 2 * pad_h - dil * (r - 1) - 1) // stride + 1
    q = (w + 2 * pad_w - dil * (s - 1) - 1) // stride + 1
    return dict(n=n, c=c, h=h, w=w, k=k, r=r, s=s, pad_h=pad_h, pad_w=pad_w, stride=stride, dil=dil, group=group,
                x_nhwc=nhwc, y_nhwc=nhwc, bias=bias, relu=relu, p=p, q=q)


def _net(case):
    """The layers of a network on square images of `side` pixels; planes shrink by halves, rounded
    up, as padded strided layers and Caffe's pooling do."""
    wl = workloads.workload(NETS[case["net"]], case["n"])
    out = []
    for l in wl.layers:
        h = l.h if case["net"] == "alexnet_pair" else -(-case["side"] // (224 // l.h))
        c = _conv(case["n"], l.c, h, h, l.k, l.r, l.r, l.pad, l.pad, l.stride, l.dil, l.group, case.get("nhwc", False), True, l.relu)
        if l.c < 8:
            c["x_nhwc"] = False  # images come as NCHW
        out.append(c)
    return out


def _layers(case):
    kind = case["kind"]
    if kind == "layer":
        return [_conv(**{k: v for k, v in case.items() if k not in ("kind", "name")})]
    if kind == "fc":
        n, c, m, k = case["n"], case["c"], case["hidden"], case["k"]
        return [_conv(n, a, 1, 1, b, 1, 1, 0, 0, 1, 1, 1, False, True, relu) for a, b, relu in ((c, m, True), (m, m, True), (m, k, False))]
    if kind == "blocks":
        return _net(dict(case, net="mobilenet_v1", nhwc=True))
    if kind == "load":
        return _net(dict(case, n=1, side=224))
    return _net(case)


def _x_shape(l):
    return (l["n"], l["h"], l["w"], l["c"]) if l["x_nhwc"] else (l["n"], l["c"], l["h"], l["w"])


def _y_shape(l):
    return (l["n"], l["p"], l["q"], l["k"]) if l["y_nhwc"] else (l["n"], l["k"], l["p"], l["q"])


def _w_shape(l):
    return (l["k"], l["c"] // l["group"], l["r"], l["s"])


def work(case):
    if case["kind"] == "bn":
        count = case["n"] * case["c"] * case["h"] * case["w"]
        return {"bytes": 4.0 * count + 8.0 * case["c"], "flops": 6.0 * count}
    layers = _layers(case)
    if case["kind"] == "load":  # FP32 weights in; folded and laid-out FP16 weights out
        return {"bytes": sum(8.0 * math.prod(_w_shape(l)) + 18.0 * l["k"] for l in layers),
                "flops": sum(2.0 * math.prod(_w_shape(l)) for l in layers)}
    elems = 0
    for i, l in enumerate(layers):
        elems += math.prod(_x_shape(l)) + math.prod(_w_shape(l)) + l["k"] * l["bias"] + math.prod(_y_shape(l))
        if case["kind"] == "blocks" and i % 2 == 1:  # a depthwise result stays inside its block
            elems -= 2 * math.prod(_y_shape(l))
    return {"bytes": 2.0 * elems,
            "flops": sum(2.0 * math.prod(_y_shape(l)) * math.prod(_w_shape(l)[1:]) for l in layers)}


def tolerance(case):
    """Outputs are binary16 (one rounding: 2^-11 relative).  Sums in another order fall on the other
    side of a rounding boundary now and then, by one unit; through a chain of layers such
    differences add up."""
    if case["kind"] in ("net", "host", "blocks"):
        return {"rel": 1e-3, "max": 2e-2}
    return {"rel": 5e-4, "max": 4e-3}


# ---- cases of the same ranges -------------------------------------------------------------------

def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_layer(rng):
    shape = rng.choice(("square", "square", "square", "pointwise", "pointwise", "depthwise", "stem", "grouped", "rect", "dilated"))
    n, h = _log(rng, 1, 64), _log(rng, 7, 224)
    w = h if rng.random() < 0.5 else _log(rng, 7, 224)
    c, k = _log(rng, 9, 1024), _log(rng, 8, 2048)
    if rng.random() < 0.6:  # most networks' widths are multiples of 16
        c, k = -(-c // 16) * 16, -(-k // 16) * 16
    stride = 2 if rng.random() < 0.25 else 1
    bias, relu = rng.random() < 0.8, rng.random() < 0.7
    nhwc = False
    r = s = 3
    dil = group = 1
    if shape == "square":
        r = s = rng.choice((3, 3, 3, 5))
        nhwc = c % 16 == 0 and rng.random() < 0.3
    elif shape == "pointwise":
        r = s = 1
        nhwc = c % 16 == 0 and rng.random() < 0.3
    elif shape == "depthwise":
        k = group = c
        nhwc = c % 8 == 0 and rng.random() < 0.4
    elif shape == "stem":
        c, k = rng.choice((1, 3, 3, 4)), 16 * rng.randint(1, 8)
        r = s = rng.choice((3, 3, 5, 7, 11))
        h, w = max(h, 32), max(w, 32)
        stride = rng.choice((1, 2, 2, 4 if r > 5 else 2))
    elif shape == "grouped":
        group = rng.choice((2, 2, 2, 4))
        c, k = -(-max(c, 64) // 64) * 64, -(-k // 64) * 64
    elif shape == "rect":
        r, s = rng.choice(((1, 7), (7, 1), (1, 3), (3, 1), (5, 3)))
    else:
        dil, stride = 2, 1
    return _layer(n, c, h, w, k, r, s, dil * (r // 2), dil * (s // 2), stride, dil, group, nhwc, bias, relu)


def draw(rng):
    cases = listed()
    most = {m: max(work(c)[m] for c in cases) for m in ("bytes", "flops")}
    over_link = max(work(c)["bytes"] for c in cases if c["kind"] == "host")
    while True:
        kind = rng.choice(("layer",) * 9 + ("net",) * 5 + ("blocks", "fc", "fc", "bn", "bn", "host", "load"))
        side = rng.choice((_log(rng, 96, 256), _log(rng, 96, 256), 224))
        if kind == "layer":
            case = _draw_layer(rng)
        elif kind == "net":
            case = dict(kind=kind, net=rng.choice(("vgg16", "mobilenet_v1", "resnet50", "resnet50", "alexnet_pair")), n=_log(rng, 1, 64),
                        side=side, nhwc=rng.random() < 0.35)
            if case["net"] == "alexnet_pair":
                case.update(side=227, nhwc=False)
        elif kind == "blocks":
            case = dict(kind=kind, n=_log(rng, 1, 32), side=side)
        elif kind == "host":
            case = dict(kind=kind, net=rng.choice(("vgg16", "mobilenet_v1", "resnet50")), n=_log(rng, 1, 4), side=side)
        elif kind == "fc":
            case = dict(kind=kind, n=_log(rng, 1, 256), c=_log(rng, 256, 25088), hidden=_log(rng, 256, 4096), k=_log(rng, 10, 1000))
        elif kind == "bn":
            case = dict(kind=kind, n=_log(rng, 1, 64), c=_log(rng, 16, 1024), h=_log(rng, 7, 224), w=_log(rng, 7, 224), stored=rng.random() < 0.4)
        else:
            case = dict(kind=kind, net=rng.choice(("vgg16", "mobilenet_v1", "resnet50")))
        got = work(case)
        if got["bytes"] <= (over_link if kind == "host" else most["bytes"]) and got["flops"] <= most["flops"]:
            return case


# ---- the passes ---------------------------------------------------------------------------------

class _Random:
    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def uniform(self, shape, lo, hi, dtype=torch.float16):
        return torch.empty(shape, dtype=dtype, device="cuda").uniform_(lo, hi, generator=self.g)

    def normal(self, shape, std, dtype=torch.float16):
        return torch.empty(shape, dtype=dtype, device="cuda").normal_(0.0, std, generator=self.g)

    def weights(self, l, dtype=torch.float16):
        shape = _w_shape(l)
        return self.normal(shape, math.sqrt(2.0 / math.prod(shape[1:])), dtype)

    def image(self, l):
        return self.uniform(_x_shape(l), -1.0 if l["c"] < 8 else 0.0, 1.0)


def _desc(l):
    flags = (hgc.HGC_FLAG_X_NHWC if l["x_nhwc"] else 0) | (hgc.HGC_FLAG_Y_NHWC if l["y_nhwc"] else 0)
    return hgc.ConvDesc(l["n"], l["c"], l["h"], l["w"], l["k"], l["r"], l["s"], l["pad_h"], l["pad_w"], l["stride"], l["stride"],
                        l["dil"], l["dil"], l["group"], flags)


def _prepare_layers(case, rnd):
    """Descriptors with workspaces and registered weights, tensors, and the calls of one pass."""
    calls, last, last_shape = [], None, None
    for l in _layers(case):
        d = hgc.ConvDesc.inner_product(l["n"], l["c"], l["k"]) if case["kind"] == "fc" else _desc(l)
        d.ensure_workspace()
        x = last if last_shape == _x_shape(l) else rnd.image(l)
        w, b = rnd.weights(l), rnd.uniform((l["k"],), -0.1, 0.1) if l["bias"] else None
        d.set_weights(w)
        y = torch.empty(_y_shape(l), dtype=torch.float16, device="cuda")
        calls.append((d, x, w, b, y, l["relu"]))
        last, last_shape = y, _y_shape(l)
    return calls


def _prepare_host(case, rnd):
    calls, last, last_shape = [], None, None
    for l in _layers(case):
        d = _desc(l)
        d.ensure_workspace(host=True)
        x = last if last_shape == _x_shape(l) else rnd.image(l).cpu().pin_memory()
        w, b = rnd.weights(l).cpu().pin_memory(), rnd.uniform((l["k"],), -0.1, 0.1).cpu().pin_memory()
        y = torch.empty(_y_shape(l), dtype=torch.float16, pin_memory=True)
        calls.append((d, x, w, b, y, l["relu"]))
        last, last_shape = y, _y_shape(l)
    return calls


def _prepare_blocks(case, rnd):
    layers = _layers(case)
    stem = dict(layers[0])
    d = _desc(stem)
    d.ensure_workspace()
    x, w, b = rnd.image(stem), rnd.weights(stem), rnd.uniform((stem["k"],), -0.1, 0.1)
    d.set_weights(w)
    y = torch.empty(_y_shape(stem), dtype=torch.float16, device="cuda")
    first, blocks = (d, x, w, b, y, stem["relu"]), []
    for dw, pw in zip(layers[1::2], layers[2::2]):
        d = hgc.DwPwDesc(dw["n"], dw["c"], dw["h"], dw["w"], pw["k"], dw["stride"], hgc.HGC_FLAG_Y_NHWC)
        d.ensure_workspace()
        w_dw, b_dw = rnd.weights(dw), rnd.uniform((dw["k"],), -0.1, 0.1)
        w_pw, b_pw = rnd.weights(pw), rnd.uniform((pw["k"],), -0.1, 0.1)
        d.set_weights(w_dw, w_pw)
        z = torch.empty(_y_shape(pw), dtype=torch.float16, device="cuda")
        blocks.append((d, y, w_dw, b_dw, w_pw, b_pw, z))
        y = z
    return first, blocks


def _prepare_load(case, rnd):
    """FP32 blobs, batch-norm statistics and scales of every layer; the FP16 copies are slices of
    one buffer, each on a 16-byte boundary."""
    layers = _layers(case)
    up = lambda v: -(-v // 8) * 8  # noqa: E731
    w16, out, bias = (torch.zeros(sum(up(v) for v in sizes), dtype=torch.float16, device="cuda")
                      for sizes in ([math.prod(_w_shape(l)) for l in layers],) * 2 + ([l["k"] for l in layers],))
    over = torch.zeros(1, dtype=torch.int64, device="cuda")
    calls, at, at_b = [], 0, 0
    for l in layers:
        shape, k = _w_shape(l), l["k"]
        size = math.prod(shape)
        d = _desc(l)
        d.ensure_workspace()
        f32 = torch.float32
        calls.append((d, rnd.weights(l, f32), w16[at:at + size].view(shape), out[at:at + size].view(shape), bias[at_b:at_b + k],
                      rnd.normal((k,), 0.5, f32), rnd.uniform((k,), 0.5, 2.0, f32), rnd.uniform((k,), 0.5, 1.5, f32), rnd.normal((k,), 0.1, f32)))
        at, at_b = at + up(size), at_b + up(k)
    return calls, over, out, bias


def _prepare_bn(case, rnd):
    shape, c = (case["n"], case["c"], case["h"], case["w"]), case["c"]
    x = rnd.normal(shape, 1.5).add_(0.25)
    mean, var = rnd.normal((c,), 0.25, torch.float32), rnd.uniform((c,), 0.5, 2.0, torch.float32)
    ws = torch.empty(hgc.batchnorm_workspace_bytes(case["n"], c, case["h"] * case["w"]), dtype=torch.uint8, device="cuda")
    return x, torch.empty_like(x), mean, var, ws


def prepare(case, seed):
    rnd = _Random(seed)
    kind = case["kind"]
    make = {"host": _prepare_host, "blocks": _prepare_blocks, "load": _prepare_load, "bn": _prepare_bn}.get(kind, _prepare_layers)
    return {"case": case, "kind": kind, "held": make(case, rnd)}


def run(state):
    kind, held = state["kind"], state["held"]
    if kind == "host":
        for d, x, w, b, y, relu in held:
            hgc.conv_forward_host(d, x, w, b, y, relu)
        return [call[4] for call in held]
    if kind == "blocks":
        (d, x, w, b, y, relu), blocks = held
        hgc.conv_forward(d, x, w, b, y, relu)
        for d, x, w_dw, b_dw, w_pw, b_pw, z in blocks:
            hgc.dwpw_forward(d, x, w_dw, b_dw, w_pw, b_pw, z, True, True)
        return [y] + [block[6] for block in blocks]
    if kind == "load":
        calls, over, out, bias = held
        for d, w32, w16, w, b, mean, var, gamma, beta in calls:
            hgc.cast_f32_to_f16(w32, w16, overflow_count=over)
            hgc.bn_fold(w16, None, mean, var, 1e-5, w, b, gamma, beta)
            d.set_weights(w)
        return {"weights": out, "bias": bias, "overflow": over}
    if kind == "bn":
        x, y, mean, var, ws = held
        hgc.batchnorm_forward(x, y, 1e-5, mean, var, ws, use_stored=state["case"]["stored"])
        return {"y": y, "mean": mean, "var": var}
    for d, x, w, b, y, relu in held:
        hgc.conv_forward(d, x, w, b, y, relu)
    return [call[4] for call in held]
