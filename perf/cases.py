"""The workloads whose speed counts for this library, as a program that uses it runs them.

Every case is a dict of plain values.  `kind` says which public entry points it goes through:

  layer    one `MaskedConvLayer.run`
  stack    a network's convolution layers one after the other, each with its own mask, called eagerly
           (`graph` false) or captured once in a CUDA graph and replayed, as a server does (`graph` true)
  block    a residual block whose intermediate stays compact: conv -> conv + shortcut
  dynamic  the previous layer's activations decide which positions are computed: mask_from_activation,
           set_mask with the device mask, run
  compact  the stand-alone kept-row list of a large mask
  masks    installing a network's masks: one score map pooled and ranked for every layer, then set_mask

Layers of a stack are independent problems (no pooling or normalisation between them), with the tensor
shapes of the networks; inputs are post-activation values, filters Kaiming-normal, biases N(0, 0.01), a mask
drops `sparsity` percent of the runs of `block` consecutive output positions.
"""
import math

import numpy as np
import torch

import paper_2309_06626_b200 as asx

# C_in, C_out, k, stride, pad, input size at 224 x 224
RESNET18 = [(3, 64, 7, 2, 3, 224)] + [(64, 64, 3, 1, 1, 56)] * 4
for _c, _h in ((64, 56), (128, 28), (256, 14)):
    RESNET18 += [(_c, 2 * _c, 3, 2, 1, _h), (2 * _c, 2 * _c, 3, 1, 1, _h // 2), (_c, 2 * _c, 1, 2, 0, _h)] + \
                [(2 * _c, 2 * _c, 3, 1, 1, _h // 2)] * 2

# the same at 640 x 640 for a detection backbone: a stem, then four stages of a down-convolution and a
# cross-stage-partial block
DETECT = [(3, 32, 3, 2, 1, 640)]
for _c, _n, _h in ((64, 1, 160), (128, 2, 80), (256, 3, 40), (512, 1, 20)):
    DETECT += [(_c // 2, _c, 3, 2, 1, 2 * _h), (_c, _c // 2, 1, 1, 0, _h), (_c, _c // 2, 1, 1, 0, _h)] + \
              [(_c // 2, _c // 2, 1, 1, 0, _h), (_c // 2, _c // 2, 3, 1, 1, _h)] * _n + [(_c, _c, 1, 1, 0, _h)]

NETS = {"resnet18": (RESNET18, 224), "detect": (DETECT, 640)}
FLAGS = {"none": 0, "relu": asx.ACT_RELU, "silu": asx.ACT_SILU}


def listed():
    return [
        # the smallest call: one 3x3 layer of one image, where launch latency and host work are everything
        dict(_layer(64, 64, 3, 1, 1, 56, 56, 1, 50, 1), name="layer_56_b1"),
        # one image through a classifier, called layer by layer from Python
        dict(_stack("resnet18", 224, 1, 30, 1), name="resnet18_b1"),
        # the same from a captured graph: what a latency-bound server runs
        dict(_stack("resnet18", 224, 1, 30, 1, graph=True), name="resnet18_b1_graph"),
        # the ordinary batch: the headline configuration, kept-row lists rebuilt in every pass
        dict(_stack("resnet18", 224, 64, 50, 4, recompact=True), name="resnet18_b64"),
        # fp32 storage (the paper's own type), at a medium batch
        dict(_stack("resnet18", 224, 16, 50, 4, dtype="f32"), name="resnet18_b16_f32"),
        # a detector's backbone: large images, many narrow and 1x1 layers, SiLU
        dict(_stack("detect", 640, 16, 40, 2, act="silu", recompact=True), name="detect_b16"),
        # one large layer, moderately sparse and nearly dense
        dict(_layer(256, 256, 3, 1, 1, 28, 28, 128, 50, 4), name="conv256_b128_s50"),
        dict(_layer(256, 256, 3, 1, 1, 28, 28, 128, 10, 1), name="conv256_b128_s10"),
        # a residual block with its intermediate compact
        {"kind": "block", "C": 64, "H": 56, "W": 56, "batch": 64, "sparsity": 50, "block": 4, "name": "block_b64"},
        # a mask that comes from the activations, new for every call
        {"kind": "dynamic", "C_in": 64, "C_out": 128, "k": 3, "H": 56, "W": 56, "batch": 32, "dead": 40, "name": "dynamic_b32"},
        # the kept-row list of a mask with one entry per lowered row of a large problem
        {"kind": "compact", "rows": 1 << 27, "sparsity": 50, "name": "compact_2e27"},
        # loading a masked network: every layer's mask from one score map
        {"kind": "masks", "net": "resnet18", "size": 224, "sparsity": 30, "name": "masks_resnet18"},
    ]


def _layer(C_in, C_out, k, stride, pad, H, W, batch, sparsity, block, dtype="bf16", act="relu", recompact=False, per_row=False):
    return dict(kind="layer", C_in=C_in, C_out=C_out, k=k, stride=stride, pad=pad, H=H, W=W, batch=batch, sparsity=sparsity,
                block=block, dtype=dtype, act=act, recompact=recompact, per_row=per_row)


def _stack(net, size, batch, sparsity, block, dtype="bf16", act="relu", recompact=False, graph=False):
    return dict(kind="stack", net=net, size=size, batch=batch, sparsity=sparsity, block=block, dtype=dtype, act=act,
                recompact=recompact, graph=graph)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: layers of every geometry that the tests and the networks have (odd sizes,
    odd channel counts among them), the two networks at other batches and image sizes, and the smaller kinds."""
    while True:
        case = _draw(rng)
        w = work(case)
        layer, f32 = case["kind"] == "layer", case.get("dtype") == "f32"
        if w["bytes"] < (4e8 if f32 else 8e8 if layer else 1.1e9) and w["flops"] < (2.9e10 if f32 else 6e10 if layer else 1.1e11):
            return case


def _draw(rng):
    sparsity, block = rng.choice((0, 10, 20, 30, 40, 50, 60, 75, 90)), rng.choice((1, 1, 2, 4, 4, 16))
    pick = rng.random()
    if pick < 0.55:
        k = rng.choice((1, 3, 3, 3, 5, 7))
        C_in, C_out = _log(rng, *rng.choice(((3, 16), (8, 64), (64, 512), (64, 512), (64, 512)))), _log(rng, 16, 512)
        if rng.random() < 0.7:      # most networks have round channel counts
            C_in, C_out = (C_in if C_in < 8 else (C_in + 31) // 32 * 32), (C_out + 31) // 32 * 32
        H = _log(rng, 7, 320)
        W = H if rng.random() < 0.7 else max(7, int(H * rng.uniform(0.6, 1.7)))
        return _layer(C_in, C_out, k, rng.choice((1, 1, 2)), k // 2, H, W, _log(rng, 1, 128), sparsity, block,
                      dtype=rng.choice(("bf16", "bf16", "bf16", "f32")), act=rng.choice(("relu", "relu", "silu", "none")),
                      recompact=rng.random() < 0.5, per_row=rng.random() < 0.15)
    if pick < 0.68:
        return _stack("resnet18", rng.choice((128, 160, 192, 224, 256)), _log(rng, 1, 64), sparsity, block,
                      dtype=rng.choice(("bf16", "bf16", "bf16", "f32")), recompact=rng.random() < 0.5, graph=rng.random() < 0.5)
    if pick < 0.79:
        return _stack("detect", rng.choice((320, 416, 480, 512, 640)), _log(rng, 1, 16), sparsity, block,
                      act=rng.choice(("silu", "silu", "relu")), recompact=rng.random() < 0.5, graph=rng.random() < 0.5)
    if pick < 0.86:
        H = rng.randint(7, 56)
        return {"kind": "block", "C": rng.choice((64, 128, 256)), "H": H, "W": H if rng.random() < 0.5 else rng.randint(7, 56),
                "batch": _log(rng, 1, 64), "sparsity": sparsity, "block": block}
    if pick < 0.93:
        return {"kind": "dynamic", "C_in": rng.choice((32, 64, 128, 256)), "C_out": rng.choice((48, 64, 128, 256)), "k": rng.choice((1, 3)),
                "H": rng.randint(7, 56), "W": rng.randint(7, 56), "batch": _log(rng, 1, 32), "dead": rng.choice((10, 25, 40, 60, 80))}
    if pick < 0.965:
        return {"kind": "compact", "rows": _log(rng, 1 << 10, 1 << 27), "sparsity": sparsity}
    net = rng.choice(("resnet18", "detect"))
    size = rng.choice((128, 160, 192, 224, 256)) if net == "resnet18" else rng.choice((320, 416, 480, 512, 640))
    return {"kind": "masks", "net": net, "size": size, "sparsity": max(5, sparsity) + rng.randint(0, 4)}


def _out(H, k, stride, pad):
    return (H + 2 * pad - k) // stride + 1


def _layers_of(case):
    """The layer problems of a 'layer' or 'stack' case."""
    if case["kind"] == "layer":
        return [case]
    table, full = NETS[case["net"]]
    keep = {k: case[k] for k in ("batch", "sparsity", "block", "dtype", "act", "recompact")}
    return [dict(_layer(ci, co, k, s, p, h * case["size"] // full, h * case["size"] // full, 1, 0, 1), **keep)
            for ci, co, k, s, p, h in table]


def _runs(rows, sparsity, block):
    """Runs of positions in a mask, and how many of them are dropped (one is always kept)."""
    nblocks = -(-rows // block)
    return nblocks, min(nblocks - 1, (sparsity * nblocks + 50) // 100)


def _mask(rng, rows, sparsity, block):
    """uint8 mask on the host: `sparsity` percent of the runs of `block` positions dropped."""
    nblocks, dropped = _runs(rows, sparsity, block)
    keep = np.ones(nblocks, np.uint8)
    keep[rng.permutation(nblocks)[:dropped]] = 0
    return np.repeat(keep, block)[:rows].copy()


def _values(gen, shape, dist, dtype):
    z = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)
    if dist == "relu":
        z.clamp_(min=0)
    elif dist == "silu":
        z = torch.nn.functional.silu(z)
    return z.to(dtype)


class _Layer:
    """One layer with its mask, filters and bias, and an input for it."""

    def __init__(self, c, gen, rng):
        dt = torch.float32 if c["dtype"] == "f32" else torch.bfloat16
        Ho, Wo = _out(c["H"], c["k"], c["stride"], c["pad"]), _out(c["W"], c["k"], c["stride"], c["pad"])
        self.layer = asx.MaskedConvLayer(c["C_in"], c["C_out"], c["k"], c["k"], c["stride"], c["pad"])
        self.layer.set_mask(_mask(rng, Ho * Wo * (c["batch"] if c["per_row"] else 1), c["sparsity"], c["block"]))
        dist = "normal" if c["C_in"] <= 4 else "silu" if c["act"] == "silu" else "relu"
        self.x = _values(gen, (c["batch"], c["H"], c["W"], c["C_in"]), dist, dt)
        std = math.sqrt(2.0 / (c["k"] * c["k"] * c["C_in"]))
        self.w = (_values(gen, (c["C_out"], c["k"], c["k"], c["C_in"]), "normal", torch.float32) * std).to(dt)
        self.b = _values(gen, (c["C_out"],), "normal", torch.float32) * 0.01
        self.flags = FLAGS[c["act"]] | (asx.RECOMPACT if c["recompact"] else 0) | (asx.F32 if c["dtype"] == "f32" else 0)

    def __call__(self):
        return self.layer.run(self.x, self.w, self.b, flags=self.flags)


class _Stack:
    def __init__(self, case, gen, rng):
        self.layers = [_Layer(c, gen, rng) for c in _layers_of(case)]
        self.graph = None
        if case.get("graph"):
            side = torch.cuda.Stream()
            side.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(side):
                self.eager()                              # the layers allocate what they keep
            torch.cuda.current_stream().wait_stream(side)
            torch.cuda.synchronize()
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph):
                self.out = self.eager()

    def eager(self):
        return [layer() for layer in self.layers]

    def __call__(self):
        if self.graph is None:
            return self.eager()
        self.graph.replay()
        return self.out


class _Block:
    def __init__(self, case, gen, rng):
        C, H, W, Nb = case["C"], case["H"], case["W"], case["batch"]
        m1, m2 = (_mask(rng, H * W, case["sparsity"], case["block"]) for _ in range(2))
        self.shape = (Nb, H, W)
        self.x = _values(gen, (Nb, H, W, C), "relu", torch.bfloat16)
        std = math.sqrt(2.0 / (9 * C))
        self.w1, self.w2 = ((_values(gen, (C, 3, 3, C), "normal", torch.float32) * std).to(torch.bfloat16) for _ in range(2))
        self.b1, self.b2 = (_values(gen, (C,), "normal", torch.float32) * 0.01 for _ in range(2))
        self.mid = torch.empty((Nb * max(1, int(m1.sum())), C), dtype=torch.bfloat16, device="cuda")
        self.y = torch.empty_like(self.x)
        self.first, self.second = (asx.MaskedConvLayer(C, C, 3, 3, 1, 1) for _ in range(2))
        self.first.set_mask(m1)
        self.second.set_mask(m2)
        self.second.set_input_mask(m1)
        self.second.set_residual(self.x)

    def __call__(self):
        Nb, H, W = self.shape
        st = int(torch.cuda.current_stream().cuda_stream)
        rc = self.first.run_raw(self.x.data_ptr(), Nb, H, W, self.w1.data_ptr(), self.b1.data_ptr(), self.mid.data_ptr(),
                                asx.ACT_RELU | asx.OUT_COMPACT, st)
        rc = rc or self.second.run_raw(self.mid.data_ptr(), Nb, H, W, self.w2.data_ptr(), self.b2.data_ptr(), self.y.data_ptr(),
                                       asx.ACT_RELU | asx.IN_COMPACT, st)
        if rc:
            raise RuntimeError("asx_run returned %d" % rc)
        return [self.mid, self.y]


class _Dynamic:
    def __init__(self, case, gen, rng):
        C, k, shape = case["C_in"], case["k"], (case["batch"], case["H"], case["W"])
        self.layer = asx.MaskedConvLayer(C, case["C_out"], k, k, 1, k // 2)
        self.x = _values(gen, shape + (C,), "relu", torch.bfloat16)
        dead = torch.rand(shape + (1,), generator=gen, device="cuda") < case["dead"] / 100.0      # positions without an active channel
        self.x.masked_fill_(dead, 0)
        self.w = (_values(gen, (case["C_out"], k, k, C), "normal", torch.float32) * math.sqrt(2.0 / (k * k * C))).to(torch.bfloat16)
        self.b = _values(gen, (case["C_out"],), "normal", torch.float32) * 0.01

    def __call__(self):
        mask = asx.mask_from_activation(self.x)
        self.layer.set_mask(mask)
        return [mask, self.layer.run(self.x, self.w, self.b)]


class _Compact:
    def __init__(self, case, gen, rng):
        rows = case["rows"]
        _, dropped = _runs(rows, case["sparsity"], 1)
        self.mask = torch.ones(rows, dtype=torch.uint8, device="cuda")
        self.mask[torch.randperm(rows, generator=gen, device="cuda")[:dropped]] = 0
        self.n = rows - dropped

    def __call__(self):
        kept, count, _ = asx.compact_mask(self.mask)
        return [kept[:self.n], count]                     # only the first `count` entries are defined


class _Masks:
    def __init__(self, case, gen, rng):
        self.score = rng.random((case["size"], case["size"]), dtype=np.float32)
        self.sparsity = case["sparsity"] / 100.0
        table, full = NETS[case["net"]]
        self.layers = []
        for ci, co, k, s, p, h in table:
            Ho = _out(h * case["size"] // full, k, s, p)
            self.layers.append((asx.MaskedConvLayer(ci, co, k, k, s, p), Ho))

    def __call__(self):
        masks = []
        for layer, Ho in self.layers:
            masks.append(asx.mask_from_scores(self.score, Ho, Ho, self.sparsity))
            layer.set_mask(masks[-1])
        return masks


KINDS = {"layer": _Stack, "stack": _Stack, "block": _Block, "dynamic": _Dynamic, "compact": _Compact, "masks": _Masks}


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return KINDS[case["kind"]](case, gen, np.random.default_rng(seed))


def run(state):
    return state()


def _conv_work(C_in, C_out, k, stride, H, W, pad, batch, sparsity, block, elem, per_row=False, out_compact=False, in_rows=None):
    P = _out(H, k, stride, pad) * _out(W, k, stride, pad)
    M = P * batch
    rows = M if per_row else P
    nblocks, dropped = _runs(rows, sparsity, block)
    kept = 1.0 - dropped / nblocks
    # a strided 1x1 reads only the pixels of its kept windows
    pixels = kept * M if k == 1 else batch * H * W if in_rows is None else in_rows
    K = k * k * C_in
    out_rows = kept * M if out_compact else M
    return {"bytes": elem * (C_in * pixels + K * C_out + C_out * out_rows) + 4 * C_out + rows, "flops": 2.0 * kept * M * K * C_out}


def work(case):
    """Input, filters, bias and mask read once, output written once, and the products of the kept rows."""
    kind = case["kind"]
    if kind in ("layer", "stack"):
        each = [_conv_work(c["C_in"], c["C_out"], c["k"], c["stride"], c["H"], c["W"], c["pad"], c["batch"], c["sparsity"], c["block"],
                           4 if c["dtype"] == "f32" else 2, c["per_row"]) for c in _layers_of(case)]
    elif kind == "block":
        C, H, W, Nb, s, b = (case[k] for k in ("C", "H", "W", "batch", "sparsity", "block"))
        first = _conv_work(C, C, 3, 1, H, W, 1, Nb, s, b, 2, out_compact=True)
        kept = first["flops"] / (18.0 * C * C)
        each = [first, _conv_work(C, C, 3, 1, H, W, 1, Nb, s, b, 2, in_rows=kept), {"bytes": 2 * C * kept, "flops": 0}]
    elif kind == "dynamic":
        M = case["batch"] * case["H"] * case["W"]
        each = [_conv_work(case["C_in"], case["C_out"], case["k"], 1, case["H"], case["W"], case["k"] // 2, case["batch"], case["dead"], 1, 2, True),
                {"bytes": M, "flops": 0}]
    elif kind == "compact":
        each = [{"bytes": case["rows"] + 4 * case["rows"] * (100 - case["sparsity"]) / 100, "flops": 0}]
    else:
        table, full = NETS[case["net"]]
        each = [{"bytes": 4 * case["size"] ** 2 + _out(h * case["size"] // full, k, s, p) ** 2, "flops": 0} for _, _, k, s, p, h in table]
    return {"bytes": sum(w["bytes"] for w in each), "flops": sum(w["flops"] for w in each)}


def tolerance(case):
    if case["kind"] in ("compact", "masks"):
        return "exact"                                    # kept-row lists and masks are whole numbers
    if case.get("dtype") == "f32":
        # products of TF32 operands are exact in fp32; what may differ is the order of an fp32 sum of up to 4608 terms
        return {"rel": 1e-4, "max": 4e-3}
    # bf16 results of fp32 sums: one rounding apart where the sums differ in their last bits
    return {"rel": 5e-3, "max": 0.05}
