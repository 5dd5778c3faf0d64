"""The work whose speed is tracked: what programs have this library do, through its public entry points.

Seven kinds of case, each with listed sizes and with ranges that `draw` samples:

  infer      a MobileNet-v1-style model on device tensors: one image at a time (latency) up to the batch of 128
             that the benchmark runs, fp32 and bfloat16 storage, launch by launch or as a graph replay, also
             the atrous variants of dense-prediction models and image sizes that are no multiple of 32
  serve      the same models from and to pinned host memory with the blocking call, any batch size
  block      one training step of a depthwise-separable block: forward, then every gradient
  conv       one training step of a 3x3 convolution with bias and relu: forward, then every gradient
  head       one step of transfer learning: a dense classifier on feature vectors, its softmax, its gradients and
             the updated weights (many small calls in a row)
  matmul     one product, or one product per leading index, with any transposes and any sizes
  residual   two 3x3 convolutions, the sum with the block's input, relu and a 3x3 / 2 max pool (forward)

Values: images and matrices uniform on [-1, 1), activations inside a network on [0, 6), He-normal filters,
small biases, as the repository's own workloads draw them, with the batch normalisation folded in.
"""
import math
import weakref

import torch

import paper_1901_05350_b200 as tfjsb

_WIDTHS = (64, 128, 128, 256, 256, 512, 512, 512, 512, 512, 512, 1024, 1024)
_STRIDES = (1, 2, 1, 2, 1, 2, 1, 1, 1, 1, 1, 2, 1)
_CLASSES = 1000

_contexts = {}


def _context():
    """One context for the process, as a program would hold it."""
    if 0 not in _contexts:
        _contexts[0] = tfjsb.Context(0)
    return _contexts[0]


# ---- the cases ---------------------------------------------------------------------------------------------


def _infer(batch, alpha=1.0, hw=224, math="tf32", output_stride=32, graph=False):
    return {"kind": "infer", "batch": batch, "alpha": alpha, "hw": hw, "math": math, "output_stride": output_stride,
            "graph": graph}


def _matmul(count, m, k, n, transpose_a=False, transpose_b=False):
    return {"kind": "matmul", "count": count, "m": m, "k": k, "n": n, "transpose_a": transpose_a, "transpose_b": transpose_b}


def listed():
    cases = [
        # one small image through the smallest model, as an interactive program does: latency of a launch chain
        ("infer_025_128_b1", _infer(1, 0.25, 128)),
        # one image through the full-size model, the step captured once and replayed
        ("infer_224_b1_graph", _infer(1, graph=True)),
        # the throughput configuration of the benchmark
        ("infer_224_b128", _infer(128)),
        # the same with filters and activations kept as bfloat16
        ("infer_224_b128_bf16", _infer(128, math="bf16")),
        # dense prediction: dilated depthwise layers at output stride 16, an image size of 16 n + 1
        ("infer_atrous_257_b8", _infer(8, hw=257, output_stride=16)),
        # a server that runs the requests that have arrived, from pinned host memory, and waits for the answer
        ("serve_224_b50", {"kind": "serve", "batch": 50, "alpha": 1.0, "hw": 224}),
        # training: an inner block of the model at 56 x 56
        ("block_56_128_b32", {"kind": "block", "batch": 32, "hw": 56, "cin": 128, "cout": 128, "stride": 1}),
        # training: a 3x3 convolution of an inner layer
        ("conv_28_128_b16", {"kind": "conv", "batch": 16, "hw": 28, "cin": 128, "cout": 128, "stride": 1}),
        # transfer learning: a new classifier of 101 classes on the model's 1024 pooled features
        ("head_1024_101_b64", {"kind": "head", "batch": 64, "features": 1024, "classes": 101}),
        # the single product that the repository's first workload names
        ("matmul_512", _matmul(1, 512, 512, 512)),
        # many small products in one call, sizes that are no multiple of anything
        ("matmul_64x199_199", _matmul(64, 199, 64, 199, transpose_b=True)),
        # forward pass of a residual block and the pooling after it
        ("residual_56_64_b32", {"kind": "residual", "batch": 32, "hw": 56, "channels": 64}),
    ]
    return [dict(c, name=name) for name, c in cases]


def _log(rng, low, high):
    """A whole number between low and high, even on the logarithm."""
    return min(high, max(low, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


_LARGEST_FLOPS = 1.4e11  # of a pass: a little below the benchmark's batch of 128
_LARGEST_BYTES = 2.5e8   # of the tensors that the training and residual cases read and write


def _draw_once(rng):
    kind = rng.choice(["infer", "infer", "infer", "serve", "block", "conv", "head", "matmul", "matmul", "residual"])
    if kind in ("infer", "serve"):
        alpha, hw = rng.choice([0.25, 0.5, 0.75, 1.0]), 32 * rng.randint(3, 7)
        batch = _log(rng, 1, 127)
        if kind == "serve":
            return {"kind": "serve", "batch": batch, "alpha": alpha, "hw": hw}
        if rng.random() < 0.25:
            return _infer(_log(rng, 1, 32), alpha, 16 * rng.randint(6, 20) + 1, "tf32", rng.choice([8, 16]), rng.random() < 0.5)
        return _infer(batch, alpha, hw, rng.choice(["tf32", "bf16"]), 32, rng.random() < 0.5)
    if kind == "block":
        cin = 8 * _log(rng, 4, 64)
        return {"kind": "block", "batch": _log(rng, 1, 64), "hw": _log(rng, 7, 112), "cin": cin, "cout": cin * rng.choice([1, 2]),
                "stride": rng.choice([1, 1, 2])}
    if kind == "conv":
        return {"kind": "conv", "batch": _log(rng, 1, 64), "hw": _log(rng, 7, 224), "cin": rng.choice([3, 8 * _log(rng, 2, 32)]),
                "cout": 8 * _log(rng, 2, 32), "stride": rng.choice([1, 1, 2])}
    if kind == "head":
        return {"kind": "head", "batch": _log(rng, 1, 256), "features": rng.choice([256, 512, 768, 1024]),
                "classes": rng.choice([_log(rng, 2, 1000), 1000])}
    if kind == "residual":
        return {"kind": "residual", "batch": _log(rng, 1, 64), "hw": _log(rng, 7, 112), "channels": 8 * _log(rng, 2, 32)}
    step = rng.choice([1, 4, 4])
    size = lambda low, high: step * _log(rng, max(1, low // step), high // step)  # noqa: E731
    ta, tb = rng.random() < 0.3, rng.random() < 0.5
    if rng.random() < 0.5:
        return _matmul(1, size(16, 4096), size(16, 4096), size(16, 4096), ta, tb)
    return _matmul(_log(rng, 2, 128), size(16, 512), size(16, 512), size(16, 512), ta, tb)


def draw(rng):
    while True:
        case = _draw_once(rng)
        w = work(case)
        # gradients, and products whose rows are no multiple of 16 bytes, are fp32 arithmetic: fewer of them in a pass
        fp32 = case["kind"] in ("block", "conv") or (case["kind"] == "matmul" and (case["k"] % 4 or case["n"] % 4))
        if w["flops"] <= (_LARGEST_FLOPS / 10 if fp32 else _LARGEST_FLOPS) and w["bytes"] <= _LARGEST_BYTES:
            return case


# ---- inputs, plans and weights -------------------------------------------------------------------------------


class _Layer:
    """One record of a layer list (the fields that Context.model reads)."""

    def __init__(self, kind, filter_hw=(1, 1), stride=1, dilation=1, act="none", out_channels=0, name=""):
        self.kind, self.filter_hw, self.strides, self.dilations = kind, filter_hw, (stride, stride), (dilation, dilation)
        self.pad, self.act, self.out_channels, self.name = "same", act, out_channels, name
        self.filter = self.bias = None


def _layer_list(alpha, output_stride):
    """Stem, thirteen depthwise-separable blocks, pool, dense.  Below the output stride the strides become dilations."""
    layers, current, rate = [_Layer("conv2d", (3, 3), 2, 1, "relu6", int(32 * alpha), "stem")], 2, 1
    for i, (width, stride) in enumerate(zip(_WIDTHS, _STRIDES), start=1):
        dilation = rate
        if stride > 1 and current >= output_stride:
            rate, stride = rate * stride, 1
        else:
            current *= stride
        layers.append(_Layer("depthwise_conv2d", (3, 3), stride, dilation, "relu6", 1, "dw%d" % i))
        layers.append(_Layer("conv2d", act="relu6", out_channels=int(width * alpha), name="pw%d" % i))
    return layers + [_Layer("global_avg_pool", name="pool"), _Layer("dense", out_channels=_CLASSES, name="dense")]


def _fill_weights(layers, channels, gen):
    for layer in layers:
        fh, fw = layer.filter_hw
        if layer.kind == "depthwise_conv2d":
            shape, fan_in, out = (fh, fw, channels, 1), fh * fw, channels
        elif layer.kind == "conv2d":
            shape, fan_in, out = (fh, fw, channels, layer.out_channels), fh * fw * channels, layer.out_channels
        elif layer.kind == "dense":
            shape, fan_in, out = (channels, layer.out_channels), channels, layer.out_channels
        else:
            continue
        layer.filter = (torch.randn(shape, generator=gen) * math.sqrt(2.0 / fan_in)).numpy()
        layer.bias = (torch.randn(out, generator=gen) * 0.01).numpy()
        channels = out
    return layers


class _State(dict):
    """What one user's program holds; a model is destroyed with it."""


def _device_values(seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    uniform = lambda *shape, low=-1.0, high=1.0: torch.rand(shape, generator=gen, device="cuda") * (high - low) + low  # noqa: E731
    normal = lambda *shape, std=1.0: torch.randn(shape, generator=gen, device="cuda") * std  # noqa: E731
    return gen, uniform, normal


def _prepare_model(case, seed, ctx):
    layers = _fill_weights(_layer_list(case["alpha"], case.get("output_stride", 32)), 3, torch.Generator().manual_seed(seed))
    if case["kind"] == "infer":
        layers.append(_Layer("softmax", name="softmax"))
    ctx.set_math(case.get("math", "tf32"))
    try:
        model = ctx.model(layers, (case["batch"], case["hw"], case["hw"], 3))
    finally:
        ctx.set_math("tf32")
    _, uniform, _ = _device_values(seed)
    state = _State(case=case, ctx=ctx, model=model, x=uniform(*model.input_shape))
    weakref.finalize(state, model.close)
    if case["kind"] == "serve":
        state["x"] = state["x"].cpu().pin_memory()
        state["out"] = torch.empty(model.output_shape).pin_memory()
    elif case["graph"]:
        state["out"] = torch.empty(model.output_shape, device="cuda")
        model.run(state["x"], out=state["out"])
        model.set_graph(True)
    return state


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    if kind in ("infer", "serve"):
        return _prepare_model(case, seed, ctx)
    gen, uniform, normal = _device_values(seed)
    s = _State(case=case, ctx=ctx)
    if kind == "matmul":
        lead = () if case["count"] == 1 else (case["count"],)
        m, k, n = case["m"], case["k"], case["n"]
        s["a"] = uniform(*lead, *((k, m) if case["transpose_a"] else (m, k)))
        s["b"] = uniform(*lead, *((n, k) if case["transpose_b"] else (k, n)))
    elif kind == "head":
        batch, features, classes = case["batch"], case["features"], case["classes"]
        s["x"] = uniform(batch, features, low=0.0, high=2.0)  # averages of relu6 outputs
        s["w"] = normal(features, classes, std=math.sqrt(2.0 / features))
        s["b"] = normal(classes, std=0.01)
        labels = torch.randint(classes, (batch,), generator=gen, device="cuda")
        s["targets"] = torch.nn.functional.one_hot(labels, classes).float()
        s["rate"] = torch.full((classes,), 0.01 / batch, device="cuda")
    elif kind == "residual":
        c = case["channels"]
        s["x"] = uniform(case["batch"], case["hw"], case["hw"], c, low=0.0, high=6.0)
        for name in ("1", "2"):
            s["f" + name] = normal(3, 3, c, c, std=math.sqrt(2.0 / (9 * c)))
            s["b" + name] = normal(c, std=0.01)
    else:
        n, hw, cin, cout = case["batch"], case["hw"], case["cin"], case["cout"]
        ho = -(-hw // case["stride"])
        image = cin == 3
        s["x"] = uniform(n, hw, hw, cin, low=-1.0 if image else 0.0, high=1.0 if image else 6.0)
        if kind == "block":
            s["fd"], s["bd"] = normal(3, 3, cin, 1, std=math.sqrt(2.0 / 9)), normal(cin, std=0.01)
            s["fp"], s["bp"] = normal(1, 1, cin, cout, std=math.sqrt(2.0 / cin)), normal(cout, std=0.01)
        else:
            s["f"], s["b"] = normal(3, 3, cin, cout, std=math.sqrt(2.0 / (9 * cin))), normal(cout, std=0.01)
        s["dy"] = normal(n, ho, ho, cout)
    return s


# ---- one pass --------------------------------------------------------------------------------------------------


def run(s):
    return _RUN[s["case"]["kind"]](s)


def _run_infer(s):
    probs = s["model"].run(s["x"], out=s.get("out"))
    return {"probs": probs, "logits": s["model"].layer_output_f32(s["model"].n_layers - 2)}


def _run_serve(s):
    return {"logits": s["model"].run_host(s["x"], s["out"])}


def _run_block(s):
    ctx, x, st = s["ctx"], s["x"], (s["case"]["stride"],) * 2
    h = ctx.depthwise_conv2d(x, s["fd"], st, "same", bias=s["bd"], act="relu6")
    y = ctx.conv2d(h, s["fp"], bias=s["bp"], act="relu6")
    dz = ctx.act_backprop(y, s["dy"], "relu6")
    dbp = ctx.bias_backprop(dz)
    dfp = ctx.conv2d_backprop_filter(h, s["fp"].shape, dz)
    dh = ctx.conv2d_backprop_input(h.shape, s["fp"], dz)
    dzd = ctx.act_backprop(h, dh, "relu6")
    dbd = ctx.bias_backprop(dzd)
    dfd = ctx.depthwise_conv2d_backprop_filter(x, s["fd"].shape, dzd, st, "same")
    dx = ctx.depthwise_conv2d_backprop_input(x.shape, s["fd"], dzd, st, "same")
    return {"y": y, "dbp": dbp, "dfp": dfp, "dbd": dbd, "dfd": dfd, "dx": dx}


def _run_conv(s):
    ctx, x, st = s["ctx"], s["x"], (s["case"]["stride"],) * 2
    y = ctx.conv2d(x, s["f"], st, "same", bias=s["b"], act="relu")
    dz = ctx.act_backprop(y, s["dy"], "relu")
    out = {"y": y, "db": ctx.bias_backprop(dz), "df": ctx.conv2d_backprop_filter(x, s["f"].shape, dz, st, "same")}
    if s["case"]["cin"] != 3:  # nothing wants the gradient of an image
        out["dx"] = ctx.conv2d_backprop_input(x.shape, s["f"], dz, st, "same")
    return out


def _run_head(s):
    ctx, x = s["ctx"], s["x"]
    logits = ctx.binary("add", ctx.matmul(x, s["w"]), s["b"])
    g = ctx.binary("sub", ctx.softmax(logits), s["targets"])
    dw = ctx.matmul(x, g, transpose_a=True)
    dx = ctx.matmul(g, s["w"], transpose_b=True)
    db = ctx.bias_backprop(g)
    w = ctx.binary("sub", s["w"], ctx.binary("mul", dw, s["rate"]))
    b = ctx.binary("sub", s["b"], ctx.binary("mul", db, s["rate"]))
    return {"logits": logits, "dw": dw, "dx": dx, "db": db, "w": w, "b": b}


def _run_matmul(s):
    call = s["ctx"].matmul if s["case"]["count"] == 1 else s["ctx"].batch_matmul
    return call(s["a"], s["b"], s["case"]["transpose_a"], s["case"]["transpose_b"])


def _run_residual(s):
    ctx, x = s["ctx"], s["x"]
    h = ctx.conv2d(x, s["f1"], bias=s["b1"], act="relu")
    h = ctx.conv2d(h, s["f2"], bias=s["b2"])
    y = ctx.bias_act(ctx.binary("add", h, x), act="relu")
    return {"y": y, "pooled": ctx.max_pool(y, (3, 3), (2, 2), "same")}


_RUN = {"infer": _run_infer, "serve": _run_serve, "block": _run_block, "conv": _run_conv, "head": _run_head,
        "matmul": _run_matmul, "residual": _run_residual}


# ---- what a pass cannot do without ---------------------------------------------------------------------------


def work(case):
    kind = case["kind"]
    if kind in ("infer", "serve"):
        n, size, c, flops = case["batch"], case["hw"], 3, 0.0
        values = n * (size * size * 3 + _CLASSES)
        weights = 0
        for layer in _layer_list(case["alpha"], case.get("output_stride", 32)):
            size = -(-size // layer.strides[0])
            if layer.kind == "depthwise_conv2d":
                flops += 18.0 * n * size * size * c
                weights += 10 * c
            elif layer.kind == "conv2d":
                taps = layer.filter_hw[0] * layer.filter_hw[1]
                flops += 2.0 * n * size * size * taps * c * layer.out_channels
                weights += (taps * c + 1) * layer.out_channels
                c = layer.out_channels
            elif layer.kind == "global_avg_pool":
                flops += float(n * size * size * c)
            else:
                flops += 2.0 * n * c * layer.out_channels
                weights += (c + 1) * layer.out_channels
        return {"bytes": 4.0 * values + (2.0 if case.get("math") == "bf16" else 4.0) * weights, "flops": flops}
    if kind == "matmul":
        b, m, k, n = case["count"], case["m"], case["k"], case["n"]
        return {"bytes": 4.0 * b * (m * k + k * n + m * n), "flops": 2.0 * b * m * k * n}
    if kind == "head":
        n, f, c = case["batch"], case["features"], case["classes"]
        return {"bytes": 4.0 * (2 * n * f + 3 * f * c + 2 * n * c + 4 * c), "flops": 6.0 * n * f * c}
    if kind == "residual":
        n, hw, c = case["batch"], case["hw"], case["channels"]
        half = -(-hw // 2)
        return {"bytes": 4.0 * (n * c * (2 * hw * hw + half * half) + 18 * c * c), "flops": 36.0 * n * hw * hw * c * c}
    n, hw, cin, cout = case["batch"], case["hw"], case["cin"], case["cout"]
    ho = -(-hw // case["stride"])
    image = kind == "conv" and cin == 3
    values = n * (hw * hw * cin * (1 if image else 2) + 2 * ho * ho * cout)
    if kind == "block":
        return {"bytes": 4.0 * (values + 2 * (10 * cin + (cin + 1) * cout)),
                "flops": float(n * ho * ho) * (3 * 18 * cin + 6 * cin * cout)}
    return {"bytes": 4.0 * (values + 2 * (9 * cin + 1) * cout), "flops": float(n * ho * ho) * (2 if image else 3) * 18 * cin * cout}


def tolerance(case):
    kind = case["kind"]
    # Through the model's layers: logits of the TF32 model are up to 1e-2 from those of the fp32 model (its operands
    # are cut to 11 significant bits), those of the bfloat16-storage model 5.5e-3 (every stored value is rounded)
    if kind in ("infer", "serve"):
        return {"rel": 2e-2, "max": 0.1}
    # One TF32 convolution is 8e-4 from 64-bit sums.  A gradient passes or not by the size of an activation: where
    # that lies within the last bits of zero or six, one value comes or goes whole, hence the largest difference
    if kind in ("block", "conv"):
        return {"rel": 3e-3, "max": 0.9}
    # Products whose rows are no multiple of 16 bytes have fp32 operands: 6e-7 from 64-bit sums, more for the longest
    if (kind == "matmul" and (case["k"] % 4 or case["n"] % 4)) or (kind == "head" and case["classes"] % 4):
        return {"rel": 1e-5, "max": 1e-4}
    # TF32 operands, fp32 sums: 7e-4 (one product) and 9e-4 (two convolutions in a row)
    return {"rel": 3e-3, "max": 0.02}
