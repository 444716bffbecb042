"""The work that users of this library have it do, as a list of timed cases.

A case is a dict of plain values. `prepare` makes what a program has in hand before the call (inputs on the GPU and
the library context it keeps), `run` makes one pass through the package's public entry points and returns every
output. The inputs have the distributions of the five benchmark configurations, made on the GPU: post-ReLU half-normal
activations, He-initialised weights, Laplace gradients masked by a ReLU derivative.

Kinds of cases:
  linear     one `dithered_linear_backward` call
  conv       one `dithered_conv_backward` call (stride 1 or 2)
  network    `network_backward` of a small feed-forward network (each layer's gradient comes from the layer above)
  layers     the layers of a larger network called one by one in backward order, as a training framework's own autograd
             calls them, dW overlapped (`DBP_DW_ASYNC`) and joined at the end
  quantize   `nsd_quantize` into the sparse structure and `nsd_decode_dense` back to one code per element
"""
import math

import torch

import paper_2004_04729_b200 as dbp

# Output channels of the 3x3 layers of VGG-16 for 32x32 inputs, stage by stage (a 2x2 max-pool ends each).
VGG16_STAGES = [(64, 64), (128, 128), (256, 256, 256), (512, 512, 512), (512, 512, 512)]
# The ResNet-50 bottleneck shapes: (input channels, output channels, height = width, kernel), stages 1 to 4.
RESNET50 = [(64, 64, 56, 1), (256, 64, 56, 1), (64, 64, 56, 3), (64, 256, 56, 1),
            (256, 128, 56, 1), (512, 128, 28, 1), (128, 128, 28, 3), (128, 512, 28, 1),
            (512, 256, 28, 1), (1024, 256, 14, 1), (256, 256, 14, 3), (256, 1024, 14, 1),
            (1024, 512, 14, 1), (2048, 512, 7, 1), (512, 512, 7, 3), (512, 2048, 7, 1)]
# Its stride-2 layers, by the size of their input.
RESNET50_STRIDED = [(128, 128, 56, 3), (256, 512, 56, 1), (256, 256, 28, 3), (512, 1024, 28, 1), (512, 512, 14, 3),
                    (1024, 2048, 14, 1)]

_contexts = {}


def _context():
    """The program's library context: one per device, kept."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = dbp.Context(dev)
    return _contexts[dev]


# ------------------------------------------------------------------------------------------------ cases


def _linear(dtype, B, N, K, scale, db=False):
    return {"kind": "linear", "dtype": dtype, "B": B, "N": N, "K": K, "scale": scale, "db": db}


def _conv(dtype, k, stride, B, Ci, Co, H, W, scale, db=False):
    """H, W: the size of X."""
    return {"kind": "conv", "dtype": dtype, "k": k, "stride": stride, "B": B, "Ci": Ci, "Co": Co, "H": H, "W": W,
            "scale": scale, "db": db}


def listed():
    return [
        # The smallest call in use: one fully-connected layer of an MNIST-sized model, where launches count.
        dict(_linear("f32", 128, 300, 784, 2.0), name="linear_f32_784to300_b128"),
        # A whole LeNet-300-100 backward pass: three dependent layers of a few microseconds each.
        {"name": "mlp_f32_784_300_100_10_b256", "kind": "network", "net": "mlp", "B": 256, "d0": 784, "d1": 300, "d2": 100,
         "d3": 10, "scale": 2.0},
        # A LeNet-5-like network: 5x5 kernels, one and six input channels, pooling, a ten-way classifier.
        {"name": "lenet5_f32_b128", "kind": "network", "net": "lenet5", "B": 128, "hw": 32, "c1": 6, "c2": 16, "d3": 10,
         "scale": 2.0},
        # A thousand-way classifier on 2048 features in fp32, with its bias gradient.
        dict(_linear("f32", 256, 1000, 2048, 2.0, db=True), name="linear_f32_2048to1000_b256"),
        # A wide fully-connected layer on many rows in bf16, the largest single contraction.
        dict(_linear("bf16", 4096, 4096, 1024, 5.0, db=True), name="linear_bf16_1024to4096_b4096"),
        # One 3x3 layer in fp32 at the size of a CIFAR network's first stage.
        dict(_conv("f32", 3, 1, 128, 64, 64, 32, 32, 2.0), name="conv3_f32_64to64_32x32_b128"),
        # Odd planes that no tile fits, more channels out than in, fp32, pointwise: a bottleneck layer trained in fp32.
        dict(_conv("f32", 1, 1, 30, 72, 136, 27, 19, 2.0, db=True), name="conv1_f32_72to136_27x19_b30"),
        # The pointwise layer with the largest gradient of the ResNet-50 set: bytes count, not flops.
        dict(_conv("bf16", 1, 1, 64, 64, 256, 56, 56, 5.0), name="conv1_bf16_64to256_56x56_b64"),
        # VGG-16 for CIFAR in fp32: thirteen 3x3 layers with folded ReLU masks, max-pool routing, the classifier.
        {"name": "vgg16_f32_b128", "kind": "layers", "net": "vgg16", "B": 128, "scale": 2.0},
        # The ResNet-50 bottleneck shapes in bf16, the package's headline benchmark: every shape once.
        {"name": "resnet50_bf16_b64", "kind": "layers", "net": "resnet50", "B": 64, "scale": 5.0},
        # The down-sampling layers of the same network (3x3 and pointwise, stride 2).
        {"name": "resnet50_strided_bf16_b64", "kind": "layers", "net": "resnet50_strided", "B": 64, "scale": 5.0},
        # Quantization by itself, to the sparse structure and back, at the size of that network's first-stage gradients.
        {"name": "nsd_sparse_bf16_12845056", "kind": "quantize", "dtype": "bf16", "n": 64 * 64 * 56 * 56, "scale": 5.0},
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _channels(rng, lo, hi):
    """Channel counts: multiples of eight in nearly every network, odd ones now and then."""
    c = _log(rng, lo, hi)
    return c if rng.random() < 0.15 else max(8, (c + 4) // 8 * 8)


def draw(rng):
    while True:
        c = _draw(rng)
        w = work(c)
        # bounded by the largest listed layer or layer set of the same data type
        f32 = c.get("dtype", "f32") == "f32"
        if c["kind"] == "layers" or (w["bytes"] <= 3e8 and w["flops"] <= (3e10 if f32 else 8e10)):
            return c


def _draw(rng):
    what = rng.random()
    if what < 0.25:
        dtype = rng.choice(["f32", "f32", "bf16"])
        top = 1024 if dtype == "f32" else 8192
        return _linear(dtype, _log(rng, 16, top), _log(rng, 10, min(top, 4096)), _channels(rng, 32, 4096),
                       rng.choice([2.0, 3.0, 5.0]), rng.random() < 0.5)
    if what < 0.60:
        dtype = rng.choice(["f32", "bf16", "bf16"])
        k, stride = rng.choice([(1, 1), (1, 1), (3, 1), (3, 1), (3, 1), (1, 2), (3, 2)])
        H = _log(rng, 4, 60)
        W = H if rng.random() < 0.7 else min(60, max(4, H + rng.randint(-H // 3, H // 3)))
        if stride == 2:
            H, W = H + H % 2, W + W % 2
        return _conv(dtype, k, stride, _log(rng, 8, 128), _channels(rng, 16, 1024), _channels(rng, 16, 1024), H, W,
                     rng.choice([2.0, 3.0, 5.0]), rng.random() < 0.3)
    if what < 0.70:
        if rng.random() < 0.6:
            return {"kind": "network", "net": "mlp", "B": _log(rng, 32, 512), "d0": _log(rng, 64, 1024),
                    "d1": _log(rng, 64, 512), "d2": _log(rng, 32, 256), "d3": rng.randint(10, 100), "scale": 2.0}
        return {"kind": "network", "net": "lenet5", "B": _log(rng, 16, 256), "hw": 4 * rng.randint(6, 9), "c1": rng.randint(4, 12),
                "c2": rng.randint(12, 32), "d3": rng.randint(10, 40), "scale": 2.0}
    if what < 0.85:
        net = rng.choice(["vgg16", "resnet50", "resnet50", "resnet50_strided"])
        return {"kind": "layers", "net": net, "B": _log(rng, 8, 127 if net == "vgg16" else 63),
                "scale": 2.0 if net == "vgg16" else rng.choice([3.0, 4.0, 5.0])}
    return {"kind": "quantize", "dtype": rng.choice(["f32", "bf16"]), "n": _log(rng, 1000, 2.4e7),
            "scale": rng.choice([2.0, 3.0, 5.0])}


# ------------------------------------------------------------------------------------------------ layers of a case


def _layers(case):
    """The layer calls of a case in forward order, as dicts of plain values (`pool`: a 2x2 max-pool follows the
    layer; `mask`: its gradient arrives unmasked, with the ReLU derivative beside it)."""
    kind = case["kind"]
    if kind in ("linear", "conv"):
        return [case]
    s, B = case["scale"], case["B"]
    out = []
    if case["net"] == "mlp":
        dims = [case["d0"], case["d1"], case["d2"], case["d3"]]
        for l in range(3):
            out.append(dict(_linear("f32", B, dims[l + 1], dims[l], s), mask=l < 2, no_dx=l == 0))
    elif case["net"] == "lenet5":
        hw, c1, c2 = case["hw"], case["c1"], case["c2"]
        out.append(dict(_conv("f32", 5, 1, B, 1, c1, hw, hw, s), mask=True, pool=True, no_dx=True))
        out.append(dict(_conv("f32", 5, 1, B, c1, c2, hw // 2, hw // 2, s), mask=True, pool=True))
        out.append(_linear("f32", B, case["d3"], c2 * (hw // 4) ** 2, s))
    elif case["net"] == "vgg16":
        c, hw = 3, 32
        for stage in VGG16_STAGES:
            for i, co in enumerate(stage):
                out.append(dict(_conv("f32", 3, 1, B, c, co, hw, hw, s), mask=True, pool=i == len(stage) - 1, no_dx=c == 3))
                c = co
            hw //= 2
        out.append(_linear("f32", B, 10, c, s))
    elif case["net"] == "resnet50":
        out += [_conv("bf16", k, 1, B, ci, co, hw, hw, s) for ci, co, hw, k in RESNET50]
    else:
        out += [_conv("bf16", k, 2, B, ci, co, hw, hw, s) for ci, co, hw, k in RESNET50_STRIDED]
    return out


def _sizes(L):
    """(elements of delta, X, W) of a layer."""
    if L["kind"] == "linear":
        return L["B"] * L["N"], L["B"] * L["K"], L["N"] * L["K"]
    return (L["B"] * L["Co"] * (L["H"] // L["stride"]) * (L["W"] // L["stride"]), L["B"] * L["Ci"] * L["H"] * L["W"],
            L["Co"] * L["Ci"] * L["k"] ** 2)


def work(case):
    """Each input read once, each output written once; two products of 2 flops per multiply-add (the gradient taken
    as dense)."""
    if case["kind"] == "quantize":
        e = 4 if case["dtype"] == "f32" else 2
        # delta in; bitmap (1 bit) and offsets (2 bytes per 32), the non-zero codes (a fifth to a tenth), the decoded codes
        nz = 0.39 / case["scale"] + 0.02
        return {"bytes": case["n"] * (e + 0.125 + 0.0625 + nz + 1.0), "flops": 0}
    nbytes = flops = 0.0
    chained = case["kind"] == "network"
    layers = _layers(case)
    for l, L in enumerate(layers):
        e = 4 if L["dtype"] == "f32" else 2
        nd, nx, nw = _sizes(L)
        dx = not L.get("no_dx")
        nbytes += nx * e + nw * 4
        if not (chained and l < len(layers) - 1):      # within a network a gradient is made and used inside the pass
            nbytes += nd * e
        if dx:
            nbytes += nw * e + nx * e
        if L.get("mask"):
            nbytes += nd
        if L.get("pool"):
            nbytes += nd / 4 + (nd * 4 if not chained else 0)
        macs = nd * (nw // (L["N"] if L["kind"] == "linear" else L["Co"]))
        flops += 2.0 * macs * (2 if dx else 1)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    if case["kind"] == "quantize":
        return {"rel": 1e-6, "differ": 1e-6}
    if case["kind"] == "network":
        # The gradient of a layer comes out of the layer above. Sums in another order differ by 1e-6, and a value that
        # sits on a rounding threshold then gets the next code: one code among some thousand.
        return {"rel": 2e-2, "max": 0.99}
    layers = _layers(case)
    # bf16 results round once (2^-9); fp32 sums (fp32 operands may enter as two bf16 pieces) agree to 1e-5
    return {"rel": 4e-3} if any(L["dtype"] == "bf16" for L in layers) else {"rel": 1e-5}


# ------------------------------------------------------------------------------------------------ inputs


class _Maker:
    def __init__(self, seed):
        self.dev = torch.device("cuda", torch.cuda.current_device())
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(int(seed))

    def normal(self, *shape, sigma=1.0):
        return torch.randn(*shape, generator=self.g, device=self.dev) * sigma

    def uniform(self, *shape):
        return torch.rand(*shape, generator=self.g, device=self.dev)

    def laplace(self, *shape, b=1.0):
        u = self.uniform(*shape) - 0.5
        return -b * torch.sign(u) * torch.log1p(-2.0 * u.abs().clamp(max=0.4999999))

    def mask(self, *shape):
        return (self.uniform(*shape) < 0.5).to(torch.uint8)


def _make_layer(m, L, with_delta=True):
    """The layer's own tensors: delta, X, W, and where it has them its ReLU mask and pooling positions."""
    dt = torch.float32 if L["dtype"] == "f32" else torch.bfloat16
    st = {"L": L}
    if L["kind"] == "linear":
        dshape = (L["B"], L["N"])
        X, W = m.uniform(L["B"], L["K"]), m.normal(L["N"], L["K"], sigma=L["K"] ** -0.5)
        b = 1e-3
    else:
        dshape = (L["B"], L["Co"], L["H"] // L["stride"], L["W"] // L["stride"])
        X = torch.relu(m.normal(L["B"], L["Ci"], L["H"], L["W"]))
        W = m.normal(L["Co"], L["Ci"], L["k"], L["k"], sigma=(2.0 / (L["Ci"] * L["k"] ** 2)) ** 0.5)
        b = 1e-4
    st["X"], st["W"] = X.to(dt), W.to(dt)
    if L.get("mask"):
        st["mask"] = m.mask(*dshape)
    if with_delta:
        d = m.laplace(*dshape, b=b)
        if not L.get("mask"):
            d = d * m.mask(*dshape)
        st["delta"] = d.to(dt)
    if L.get("pool"):
        # the routing of the gradient that arrives at the pooled output
        shape = (dshape[0], dshape[1], dshape[2] // 2, dshape[3] // 2)
        st["argmax"] = torch.randint(0, 4, shape, generator=m.g, device=m.dev, dtype=torch.int8)
    return st


def prepare(case, seed):
    m = _Maker(seed)
    state = {"case": case, "ctx": _context(), "seed": int(seed)}
    if case["kind"] == "quantize":
        d = m.laplace(case["n"], b=1e-4) * m.mask(case["n"])
        state["delta"] = d.to(torch.float32 if case["dtype"] == "f32" else torch.bfloat16)
        state["sparse"] = dbp.SparseGradient(case["n"], state["ctx"].device)      # kept and written again by every pass
        return state
    layers = _layers(case)
    if case["kind"] != "network":
        state["layers"] = [_make_layer(m, L) for L in layers]
        return state
    made = [_make_layer(m, L, with_delta=False) for L in layers]
    state["kinds"] = [L["kind"] for L in layers]
    state["Xs"] = [s["X"] for s in made]
    state["Ws"] = [s["W"] for s in made]
    state["masks"] = [s.get("mask") for s in made]
    state["argmax"] = [s.get("argmax") for s in made]
    # softmax minus one-hot on random labels, averaged over the batch
    B, n = case["B"], case["d3"]
    p = torch.softmax(m.normal(B, n), dim=1)
    labels = torch.randint(0, n, (B,), generator=m.g, device=m.dev)
    p[torch.arange(B, device=m.dev), labels] -= 1.0
    state["delta_out"] = p / B
    return state


# ------------------------------------------------------------------------------------------------ one pass


def _call(ctx, st, seed, flags=0):
    L = st["L"]
    if L["kind"] == "linear":
        return dbp.dithered_linear_backward(ctx, st["delta"], st["X"], st["W"], seed, L["scale"], need_db=L["db"], flags=flags)
    return dbp.dithered_conv_backward(ctx, st["delta"], st["X"], st["W"], seed, L["scale"], need_db=L["db"],
                                      need_dX=not L.get("no_dx"), flags=flags, stride=L["stride"])


def run(state):
    ctx, case, seed = state["ctx"], state["case"], state["seed"]
    if case["kind"] == "quantize":
        q = dbp.nsd_quantize(ctx, state["delta"], seed, case["scale"], out=state["sparse"])
        return {"codes": dbp.nsd_decode_dense(ctx, q), "bitmap": q.bitmap, "offsets": q.offsets, "Delta": q.delta, "nnz": q.nnz}
    if case["kind"] == "network":
        res = dbp.network_backward(ctx, state["kinds"], state["Xs"], state["Ws"], state["masks"], state["argmax"],
                                   state["delta_out"], case["scale"], seed, with_sparse=False, flags=dbp.DBP_DW_ASYNC)
        ctx.join()
        return res
    layers = state["layers"]
    if len(layers) == 1:
        return _call(ctx, layers[0], seed)
    out = [None] * len(layers)
    for l in range(len(layers) - 1, -1, -1):
        st = layers[l]
        r = {}
        if "argmax" in st:                                 # the gradient above the pool goes through its routing
            above = out[l + 1]["dX"].view(st["argmax"].shape)
            r["routed"] = dbp.maxpool2x2_backward(ctx, above, st["argmax"])
        if "mask" in st:
            ctx.set_relu_mask(st["mask"])
        r.update(_call(ctx, st, dbp.layer_seed(seed, l), flags=dbp.DBP_DW_ASYNC))
        out[l] = r
    ctx.join()
    return out
