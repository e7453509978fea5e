"""The work a user of the library has it do, as measurable cases.

An inference program calls single operators (Conv with constant or with per-call weights, depthwise
Conv, Gemm) and whole chained models (the MNIST network, ResNet-50 v1) through
``paper_2008_08272_b200.binding`` and ``paper_2008_08272_b200.resnet50_chain``.  A case is a dict of
plain values; ``listed()`` gives the fixed ones, ``draw(rng)`` one more of the same ranges.

Keys by ``op``:
  conv      batch, channels, height, width, filters, kernel, stride, dilation, group, pad, bias, relu,
            residual (an addend of the output's shape, fused), weights: "constant" (packed once, run from
            the copy, output and workspace buffers kept, as resnet50_chain.py does) or "per_call"
            (the plain run call, which allocates its output)
  gemm      M, N, K, transA, transB, C ("none", "scalar", "row" = (N,), "column" = (M, 1), "full"), alpha,
            beta, relu
  mnist     batch
  resnet50  batch
"""
import math

import torch

from paper_2008_08272_b200 import binding
from paper_2008_08272_b200.resnet50_chain import Resnet50Chain


def _conv(name, x, w, **kw):
    c = {"name": name, "op": "conv", "batch": x[0], "channels": x[1], "height": x[2], "width": x[3], "filters": w[0],
         "kernel": w[1], "stride": 1, "dilation": 1, "group": 1, "pad": 0, "bias": True, "relu": True,
         "residual": False, "weights": "constant"}
    c.update(kw)
    return c


def _gemm(name, M, N, K, **kw):
    c = {"name": name, "op": "gemm", "M": M, "N": N, "K": K, "transA": False, "transB": False, "C": "row",
         "alpha": 1.0, "beta": 1.0, "relu": False}
    c.update(kw)
    return c


def listed():
    return [
        # The smallest model, one image at a time: five operator calls of a few microseconds each (latency).
        {"name": "mnist_b1", "op": "mnist", "batch": 1},
        # A classifier head behind it: the smallest single Gemm call (configuration 2 of the benchmark spec).
        _gemm("gemm_head_64x10x256", 64, 10, 256, transB=True),
        # A dense layer of ordinary size.
        _gemm("gemm_1024", 1024, 1024, 1024, transB=True, relu=True),
        # A large dense layer with both operands as stored.
        _gemm("gemm_4096", 4096, 4096, 4096),
        # A dense layer whose sizes are no multiples of anything, A stored transposed.
        _gemm("gemm_ragged_1001x1530x777", 1001, 1530, 777, transA=True, C="column", alpha=0.5, beta=-1.5),
        # ResNet-50's stem, batch 32 (configuration 4): three input channels, 7x7, stride 2.
        _conv("conv_stem_b32", (32, 3, 224, 224), (64, 7), stride=2, pad=3),
        # ResNet-50 stage 2, batch 32 (configuration 3): the ordinary 3x3.
        _conv("conv_3x3_b32", (32, 64, 56, 56), (64, 3), pad=1),
        # A down-sampling projection, batch 32 (configuration 4): strided 1x1.  Weights of the call, not constants.
        _conv("conv_proj_1x1_s2_b32", (32, 256, 56, 56), (512, 1), stride=2, weights="per_call"),
        # The depthwise layer of configuration 5 at batch 64.
        _conv("conv_depthwise_b64", (64, 256, 28, 28), (256, 3), pad=1, group=256),
        # An image of odd size through a dilated, grouped layer with a residual addend, weights of the call.
        _conv("conv_dilated_grouped_odd", (4, 96, 75, 61), (192, 3), pad=2, dilation=2, group=2, residual=True,
              weights="per_call"),
        # ResNet-50 v1 end to end: one image (latency and host work count) ...
        {"name": "resnet50_b1", "op": "resnet50", "batch": 1},
        # ... and the batch the benchmark is quoted on (the largest case).
        {"name": "resnet50_b64", "op": "resnet50", "batch": 64},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _channels(rng, lo, hi):
    """Channel counts as networks have them: mostly multiples of 16, sometimes any number."""
    c = _log_int(rng, lo, hi)
    return c if c < 16 or rng.random() < 0.25 else (c + 8) // 16 * 16


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    while True:
        kind = rng.choice(("conv",) * 4 + ("conv1x1",) * 3 + ("depthwise",) * 2 + ("gemm",) * 5 + ("resnet50",) * 2 + ("mnist",))
        if kind == "mnist":
            return {"op": "mnist", "batch": _log_int(rng, 2, 256)}
        if kind == "resnet50":
            return {"op": "resnet50", "batch": _log_int(rng, 2, 48)}
        if kind == "gemm":
            c = _gemm("", _log_int(rng, 16, 6000), _log_int(rng, 10, 6000), _log_int(rng, 24, 6000),
                      transA=rng.random() < 0.3, transB=rng.random() < 0.5,
                      C=rng.choice(("none", "row", "row", "row", "column", "full", "scalar")),
                      alpha=rng.choice((1.0, 1.0, 0.5)), beta=rng.choice((1.0, 1.0, -1.5)), relu=rng.random() < 0.5)
            if rng.random() < 0.6:          # layer widths as networks have them
                for d in ("M", "N", "K"):
                    c[d] = max(16, (c[d] + 8) // 16 * 16)
        else:
            k = 1 if kind == "conv1x1" else rng.choice((3, 3, 3, 5, 7) if kind == "conv" else (3, 3, 5))
            side = _log_int(rng, 7, 224)
            h, w = (side, side) if rng.random() < 0.6 else (side, max(5, int(side * rng.uniform(0.6, 1.6))))
            stride = 2 if rng.random() < (0.5 if k == 7 else 0.25) else 1
            dilation = 2 if k == 3 and stride == 1 and rng.random() < 0.1 else 1
            chan = _channels(rng, 32, 2048) if k == 1 else 3 if k == 7 and rng.random() < 0.5 else _channels(rng, 8, 512)
            filt, group = _channels(rng, 16, 2048 if k == 1 else 512), 1
            if kind == "depthwise":
                filt = group = chan
            elif kind == "conv" and chan % 32 == 0 and filt % 4 == 0 and rng.random() < 0.15:
                group = rng.choice((2, 4))
            c = _conv("", (_log_int(rng, 1, 64), chan, h, w), (filt, k), stride=stride, dilation=dilation, group=group,
                      pad=dilation * (k - 1) // 2, bias=rng.random() < 0.9, relu=rng.random() < 0.8,
                      residual=rng.random() < 0.2, weights=rng.choice(("constant", "constant", "per_call")))
        need = work(c)
        # from the smallest calls up to a good part of the largest listed case
        if 2e6 <= need["flops"] <= 2e10 and need["bytes"] <= 5e8:
            del c["name"]
            return c


# --------------------------------------------------------------------- shapes
def _conv_shapes(c):
    ext = (c["kernel"] - 1) * c["dilation"] + 1
    p, q = ((s + 2 * c["pad"] - ext) // c["stride"] + 1 for s in (c["height"], c["width"]))
    x = (c["batch"], c["channels"], c["height"], c["width"])
    w = (c["filters"], c["channels"] // c["group"], c["kernel"], c["kernel"])
    return x, w, (c["batch"], c["filters"], p, q)


_C_SHAPES = {"none": lambda m, n: None, "scalar": lambda m, n: (), "row": lambda m, n: (n,), "column": lambda m, n: (m, 1),
             "full": lambda m, n: (m, n)}

# The MNIST network of the ONNX Model Zoo: 5x5 -> pool 2 -> 5x5 -> pool 3 -> dense.
_MNIST_CONVS = (((1, 28), (8, 1, 5, 5)), ((8, 14), (16, 8, 5, 5)))
_RESNET50_WEIGHTS = 25_530_472          # 53 convolutions' weights and biases and the 2048 x 1000 head
_RESNET50_FLOPS_PER_IMAGE = 7_715_946_496


def work(case):
    """Each input read once, each output written once; multiply-adds counted as two, taps on padding included."""
    if case["op"] == "conv":
        x, w, y = _conv_shapes(case)
        ny = math.prod(y)
        nx = math.prod(x)
        if case["kernel"] == 1 and case["stride"] > 1:      # skipped rows need not be read
            nx = nx // case["height"] * -(-case["height"] // case["stride"])
        n = nx + math.prod(w) + ny * (2 if case["residual"] else 1) + (w[0] if case["bias"] else 0)
        return {"bytes": 4 * n, "flops": 2 * ny * w[1] * w[2] * w[3]}
    if case["op"] == "gemm":
        m, n, k = case["M"], case["N"], case["K"]
        cs = _C_SHAPES[case["C"]](m, n)
        return {"bytes": 4 * (m * k + k * n + m * n + (math.prod(cs) if cs is not None else 0)), "flops": 2 * m * n * k}
    b = case["batch"]
    if case["op"] == "mnist":
        return {"bytes": 4 * (b * (784 + 10) + 200 + 8 + 3200 + 16 + 2560 + 10),
                "flops": 2 * b * (8 * 784 * 25 + 16 * 196 * 200 + 2560)}
    return {"bytes": 4 * (b * (3 * 224 * 224 + 1000) + _RESNET50_WEIGHTS), "flops": b * _RESNET50_FLOPS_PER_IMAGE}


def tolerance(case):
    """Operands of the tensor-core paths carry TF32's 10-bit mantissa (2^-11 each); depthwise and thin
    contractions, and Gemms whose rows are no multiples of 16 bytes, are fp32 throughout."""
    fp32, tf32 = {"rel": 1e-5}, {"rel": 1e-3}
    if case["op"] == "resnet50":            # 54 TF32 layers in a row
        return {"rel": 1e-2}
    if case["op"] == "mnist":
        return fp32
    if case["op"] == "conv":
        k = case["channels"] // case["group"] * case["kernel"] ** 2
        return fp32 if k < 32 or case["group"] == case["channels"] else tf32
    rows = (case["M"] if case["transA"] else case["K"], case["K"] if case["transB"] else case["N"])
    return fp32 if case["K"] < 32 or any(r % 4 for r in rows) else tf32


# --------------------------------------------------------------------- states
class _Draws:
    """Seeded values on the GPU."""

    def __init__(self, seed):
        self.dev = torch.device("cuda:0")
        self.g = torch.Generator(device=self.dev)
        self.g.manual_seed(seed)

    def uniform(self, *shape):              # activations behind a Relu
        return torch.rand(shape, generator=self.g, device=self.dev)

    def normal(self, *shape, std=1.0):
        return torch.randn(shape, generator=self.g, device=self.dev) * std

    def weights(self, *shape):              # He-normal
        return self.normal(*shape, std=math.sqrt(2.0 / math.prod(shape[1:])))


def prepare(case, seed):
    d = _Draws(seed)
    if case["op"] == "resnet50":
        b = case["batch"]
        return {"op": "resnet50", "x": d.uniform(b, 3, 224, 224), "net": Resnet50Chain(b, d.dev, seed=seed)}
    if case["op"] == "mnist":
        b = case["batch"]
        s = {"op": "mnist", "b": b, "x": d.normal(b, 1, 28, 28), "layers": []}
        for (c, hw), w in _MNIST_CONVS:
            desc = binding.Conv2dDesc((b, c, hw, hw), w, pads=(2, 2, 2, 2), has_bias=True, fuse_relu=True)
            wt = d.weights(*w)
            s["layers"].append((desc, wt, desc.prepack(wt), d.normal(w[0], std=0.1)))
        s["fc"] = (d.normal(256, 10, std=1.0 / 16), d.normal(10, std=0.1))
        return s
    if case["op"] == "gemm":
        m, n, k = case["M"], case["N"], case["K"]
        cs = _C_SHAPES[case["C"]](m, n)
        return {"op": "gemm", "A": d.normal(*((k, m) if case["transA"] else (m, k))),
                "B": d.normal(*((n, k) if case["transB"] else (k, n))), "C": None if cs is None else d.normal(*cs),
                "kw": {"alpha": case["alpha"], "beta": case["beta"], "transA": case["transA"], "transB": case["transB"],
                       "fuse_relu": case["relu"]}}
    x, w, y = _conv_shapes(case)
    s = {"op": "conv", "X": d.uniform(*x), "W": d.weights(*w), "B": d.normal(w[0], std=0.01) if case["bias"] else None,
         "R": d.normal(*y) if case["residual"] else None}
    s["desc"] = binding.Conv2dDesc(x, w, pads=(case["pad"],) * 4, strides=(case["stride"],) * 2,
                                   dilations=(case["dilation"],) * 2, group=case["group"], has_bias=case["bias"],
                                   fuse_relu=case["relu"])
    s["packed"] = None
    if case["weights"] == "constant":
        s["packed"] = s["desc"].prepack(s["W"])
        s["Y"] = torch.empty(y, device=d.dev)
        s["ws"] = torch.empty(max(16, s["desc"].workspace_bytes), dtype=torch.uint8, device=d.dev)
    return s


def run(s):
    if s["op"] == "resnet50":
        return s["net"].forward(s["x"])
    if s["op"] == "mnist":
        t = s["x"]
        for (desc, w, packed, b), pool in zip(s["layers"], (2, 3)):
            t = binding.onnx_maxpool2d(desc.run_prepacked(t, w, packed, b), (pool, pool), strides=(pool, pool))
        return binding.onnx_matmul_add(t.view(s["b"], 256), *s["fc"])
    if s["op"] == "gemm":
        return binding.onnx_gemm(s["A"], s["B"], s["C"], **s["kw"])
    if s["packed"] is not None:
        return s["desc"].run_prepacked(s["X"], s["W"], s["packed"], s["B"], s["R"], Y=s["Y"], workspace=s["ws"])
    if s["R"] is not None:
        return s["desc"].run_add(s["X"], s["W"], s["B"], s["R"])
    return s["desc"].run(s["X"], s["W"], s["B"])
