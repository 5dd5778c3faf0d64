"""GPU parity of the ops beyond the MobileNet path: maxPool, elementwise add / sub / mul, rank-3 matMul,
dilated depthwise convolution and the atrous (output stride 16 / 8) MobileNet variants built from it.

Tolerances.  maxPool selects an input value and add / sub / mul are one correctly rounded fp32
operation per element, so both must match the oracle bit for bit (NaNs in the same places).  A
rank-3 matMul is one rank-2 product per leading index through the same kernels as tfjsb_matmul:
relative Frobenius error <= 5e-3 against the exact oracle on the tensor cores, <= 1e-5 in fp32 mode,
bit-identical on small integers.
"""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import dev, host, rel_fro, same_bits

pytestmark = pytest.mark.gpu

POOL_CASES = [
    # N, H, W, C, window, strides, pad
    (2, 112, 112, 32, (3, 3), (2, 2), "same"),    # even size, stride 2: padding after only
    (1, 7, 7, 1024, (7, 7), (1, 1), "valid"),     # global
    (3, 13, 17, 5, (2, 3), (2, 1), "valid"),      # unequal window and strides, odd channel count
    (1, 9, 9, 8, (3, 3), (1, 1), "same"),
    (1, 1, 1, 4, (3, 3), (1, 1), "same"),         # window mostly outside the image
    (2, 33, 20, 64, (5, 5), (3, 3), "same"),
]


def same_bits_or_both_nan(a, b):
    a, b = np.ascontiguousarray(a, np.float32), np.ascontiguousarray(b, np.float32)
    nan = np.isnan(a)
    return a.shape == b.shape and np.array_equal(nan, np.isnan(b)) and np.array_equal(a[~nan].view(np.uint32), b[~nan].view(np.uint32))


@pytest.mark.parametrize("case", POOL_CASES)
def test_max_pool_bit_exact(ctx, oracle, case):
    N, H, W, C, k, s, pad = case
    x = si.normal(501, 0, (N, H, W, C), -1, 2)   # mostly negative: zero padding would win wrongly
    got = host(ctx.max_pool(dev(x), k, s, pad))
    want = oracle.max_pool(x, k, s, pad)
    assert got.shape == want.shape and same_bits(got, want)
    x.reshape(-1)[::97] = np.nan                  # NaNs reach exactly the windows that contain them
    assert same_bits_or_both_nan(host(ctx.max_pool(dev(x), k, s, pad)), oracle.max_pool(x, k, s, pad))


def test_max_pool_rejects_bad_arguments(ctx, tfjsb):
    import torch

    x = torch.zeros(1, 4, 4, 4, device="cuda")
    with pytest.raises(tfjsb.TfjsbError) as err:
        ctx.max_pool(x, (5, 5), (1, 1), "valid")                       # window larger than the image
    assert err.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError):
        ctx.max_pool(x, (2, 2), (2, 2), "valid", out=torch.zeros(1, 3, 3, 4, device="cuda"))  # wrong out shape


BINARY_SHAPES = [(4, 56, 56, 64), (3, 5, 7, 6), (1000,), (2, 3, 5), (1, 1, 1, 4), (128, 1000), (7, 13, 3)]


@pytest.mark.parametrize("op", ["add", "sub", "mul"])
@pytest.mark.parametrize("shape", BINARY_SHAPES)
def test_binary_ops_bit_exact(ctx, oracle, op, shape):
    a = si.normal(502, 0, shape, 0, 10)
    b = si.normal(502, 1, shape, 0, 10)
    v = si.normal(502, 2, (shape[-1],), 0, 10)
    a.reshape(-1)[::53] = np.nan
    b.reshape(-1)[::71] = np.inf
    assert same_bits_or_both_nan(host(ctx.binary(op, dev(a), dev(b))), oracle.binary(op, a, b))
    assert same_bits_or_both_nan(host(ctx.binary(op, dev(a), dev(v))), oracle.binary(op, a, v))


def test_binary_rejects_bad_arguments(ctx, tfjsb):
    import torch

    a = torch.zeros(2, 8, device="cuda")
    with pytest.raises(tfjsb.TfjsbError) as err:
        ctx.binary("add", a, torch.zeros(2, 4, device="cuda"))
    assert err.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as err:
        ctx.binary("add", a, torch.zeros(8, device="cuda"), out=a)     # out aliases an input
    assert err.value.status_name == "INVALID_ARG"
    assert ctx.binary("mul", torch.zeros(0, 8, device="cuda"), torch.zeros(8, device="cuda")).shape == (0, 8)


BATCH_MATMUL_CASES = [
    # B, M, K, N, transpose_a, transpose_b
    (4, 128, 64, 64, False, False),
    (3, 300, 100, 72, False, True),
    (2, 49, 1024, 256, True, False),     # few tiles, long K: each product is cut along K
    (5, 9, 13, 5, False, False),         # slices not 16-byte aligned: CUDA-core kernel
    (1, 512, 512, 512, True, True),
    (70, 68, 36, 100, True, False),      # both operands transposed in one launch each, ragged 32 x 32 tiles
]


@pytest.mark.parametrize("case", BATCH_MATMUL_CASES)
def test_batch_matmul_parity(ctx, oracle, case):
    B, M, K, N, ta, tb = case
    a = si.uniform(503, 0, (B, K, M) if ta else (B, M, K), -1, 1)
    b = si.uniform(503, 1, (B, N, K) if tb else (B, K, N), -1, 1)
    got = host(ctx.batch_matmul(dev(a), dev(b), ta, tb))
    ctx.check_device_status()
    want = oracle.batch_matmul(a, b, ta, tb)
    assert got.shape == (B, M, N)
    for i in range(B):  # per product, so that one bad slice cannot hide among good ones
        assert rel_fro(got[i], want[i]) <= 5e-3
    ai = si.small_integers(504, 0, a.shape, -8, 8)
    bi = si.small_integers(504, 1, b.shape, -8, 8)
    assert same_bits(host(ctx.batch_matmul(dev(ai), dev(bi), ta, tb)), oracle.batch_matmul(ai, bi, ta, tb))
    ctx.set_math("fp32")
    try:
        got32 = host(ctx.batch_matmul(dev(a), dev(b), ta, tb))
    finally:
        ctx.set_math("tf32")
    assert rel_fro(got32, want) <= 1e-5


def test_batch_matmul_rejects_bad_arguments(ctx, tfjsb):
    import torch

    with pytest.raises(tfjsb.TfjsbError) as err:
        ctx.batch_matmul(torch.zeros(2, 4, 8, device="cuda"), torch.zeros(3, 8, 4, device="cuda"))
    assert err.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as err:
        ctx.batch_matmul(torch.zeros(2, 4, 8, device="cuda"), torch.zeros(2, 7, 4, device="cuda"))
    assert err.value.status_name == "SHAPE"


DILATED_DW_CASES = [
    # N, H, W, C, dilation: 3x3 depthwise, stride 1, 'same' (the atrous layers of output-stride-16 / -8 models)
    (2, 14, 14, 512, 2),
    (1, 28, 28, 256, 4),
    (3, 9, 11, 32, 2),     # image barely larger than the dilated window
    (1, 5, 5, 8, 4),       # dilated window larger than the image: most taps fall outside
    (2, 14, 14, 6, 2),     # channel count not a multiple of 4: the general kernel
]


@pytest.mark.parametrize("case", DILATED_DW_CASES)
def test_dilated_depthwise_parity(ctx, oracle, case):
    N, H, W, C, d = case
    x = si.uniform(505, 0, (N, H, W, C), 0, 6)
    f = si.normal(505, 1, (3, 3, C, 1), 0, 0.47)
    b = si.normal(505, 2, (C,), 0, 0.5)
    got = host(ctx.depthwise_conv2d(dev(x), dev(f), (1, 1), "same", (d, d), dev(b), "relu6"))
    want = oracle.depthwise_conv2d(x, f, (1, 1), "same", (d, d), b, "relu6")
    assert got.shape == want.shape and rel_fro(got, want) <= 1e-6
    xi = si.small_integers(506, 0, x.shape, -8, 8)
    fi = si.small_integers(506, 1, f.shape, -8, 8)
    assert same_bits(host(ctx.depthwise_conv2d(dev(xi), dev(fi), (1, 1), "same", (d, d))),
                     oracle.depthwise_conv2d(xi, fi, (1, 1), "same", (d, d)))


@pytest.mark.parametrize("output_stride", [16, 8])
def test_atrous_mobilenet_every_layer(ctx, oracle, output_stride):
    """alpha 0.25, 96x96 input, batch 2, output stride 16 / 8: every layer's output against the oracle."""
    x, layers = si.config_mobilenet_atrous(0.25, 96, 2, output_stride, seed=4243, classes=100)
    dilations = sorted({l.dilations[0] for l in layers if l.kind == "depthwise_conv2d"})
    assert dilations == ([1, 2] if output_stride == 16 else [1, 2, 4])
    want = oracle.run_model(layers, x, keep_all=True)
    assert want[-4].shape[1] == 96 // output_stride          # spatial size of the last block's output
    model = ctx.model(layers, x.shape)
    model.set_keep_all(True)
    probs = host(model.run(dev(x)))
    ctx.check_device_status()
    for i, layer in enumerate(layers):
        got = host(model.layer_output(i)) if i < len(layers) - 1 else probs
        assert got.shape == want[i].shape, layer.name
        assert rel_fro(got, want[i]) <= 2e-2, f"layer {i} ({layer.name}) diverges: {rel_fro(got, want[i]):.3e}"
    span = float(want[-2].max() - want[-2].min())
    assert np.max(np.abs(host(model.layer_output(len(layers) - 2)) - want[-2])) <= 1e-2 * span
    model.set_keep_all(False)
    assert same_bits(host(model.run(dev(x))), probs)          # the ping-pong run gives the same bits
    model.close()


@pytest.mark.parametrize("call", ["tfjsb_matmul", "tfjsb_conv2d", "tfjsb_bias_backprop", "tfjsb_run_model"])
def test_a_call_that_fails_is_not_made_twice(ctx, tfjsb, monkeypatch, call):
    """A failing call may have enqueued a part of its work (a model its first layers, a convolution the packing of its
    filter): the error that the library reports is raised, and the call is not repeated through ctypes."""
    import torch

    def repeated(*args):
        raise AssertionError("the call was made a second time")

    monkeypatch.setattr(tfjsb.lib, call, repeated)
    wrong = torch.zeros(3, 3, device="cuda")
    x, layers = si.config_mobilenet(0.25, 32, 1, seed=5, classes=10)
    model = ctx.model(layers, x.shape)
    with pytest.raises(tfjsb.TfjsbError) as e:
        if call == "tfjsb_matmul":
            ctx.matmul(torch.zeros(8, 8, device="cuda"), torch.zeros(8, 12, device="cuda"), out=wrong)
        elif call == "tfjsb_conv2d":
            ctx.conv2d(torch.zeros(1, 8, 8, 16, device="cuda"), torch.zeros(3, 3, 16, 8, device="cuda"), out=torch.zeros(1, 8, 8, 9, device="cuda"))
        elif call == "tfjsb_bias_backprop":
            ctx.bias_backprop(torch.zeros(4, 8, device="cuda"), out=torch.zeros(7, device="cuda"))
        else:
            model.run(dev(x), out=wrong)
    assert e.value.status_name == "SHAPE" and str(e.value)
    model.close()


def test_op_calls_one_after_another_see_each_others_results(ctx):
    """Each kernel is launched while the one before drains and waits for it before it reads or writes anything: chains of
    dependent small and large calls through two buffers, and calls that overwrite what the call before reads."""
    import torch

    one = {n: torch.ones(n, device="cuda") for n in (64, 1 << 20)}
    for n, o in one.items():
        bufs = [torch.zeros(n, device="cuda") for _ in range(2)]
        for i in range(200):
            ctx.binary("add", bufs[i % 2], o, out=bufs[(i + 1) % 2])
        assert float(bufs[0].min()) == 200.0 == float(bufs[0].max())
    x, w = torch.ones(256, 64, device="cuda"), torch.ones(64, 256, device="cuda")
    y, z = torch.empty(256, 256, device="cuda"), torch.empty(256, 256, device="cuda")
    for i in range(50):
        ctx.matmul(x, w, out=y)                                # 64 everywhere ...
        ctx.binary("mul", y, y, out=z)                         # ... squared
        total = ctx.bias_backprop(z)
    ctx.check_device_status()
    assert float(z.min()) == 4096.0 == float(z.max())
    assert float(total.min()) == 256 * 4096.0 == float(total.max())


@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("shape", [(64, 1024, 101), (300, 36, 65), (8, 19, 1003)])
def test_unaligned_products_between_updates_of_their_operand(ctx, shape, tb):
    """Operands that are written again and again, two buffers in turn: a product's blocks may be on an SM that has read the
    older values of its buffer, and all the same the bits are those of calls with a synchronisation after each."""
    import torch

    m, k, n = shape
    x, step = torch.rand(m, k, device="cuda"), torch.rand(n, k, device="cuda") if tb else torch.rand(k, n, device="cuda")
    first = torch.rand_like(step)

    def calls(wait):
        w, out = [first.clone(), torch.empty_like(first)], torch.empty(100, m, n, device="cuda")
        torch.cuda.synchronize()
        for i in range(100):
            ctx.matmul(x, w[i % 2], transpose_b=tb, out=out[i])
            if wait:
                torch.cuda.synchronize()
            ctx.binary("sub", w[i % 2], step, out=w[(i + 1) % 2])
            if wait:
                torch.cuda.synchronize()
        return out

    want = calls(True)
    for _ in range(3):
        assert torch.equal(calls(False), want)
    ctx.check_device_status()


def test_op_calls_captured_on_two_streams_that_join(ctx):
    import torch

    x, w, b = torch.rand(64, 96, device="cuda"), torch.rand(96, 40, device="cuda"), torch.rand(40, device="cuda")

    def work(side):
        main = torch.cuda.current_stream()
        z = torch.zeros(64, 40, device="cuda")
        a = ctx.binary("add", ctx.matmul(x, w), b)
        z.add_(a)                                              # another library's kernel in between
        side.wait_stream(main)
        with torch.cuda.stream(side):
            s = ctx.bias_act(ctx.binary("mul", z, a), act="relu6")
        c = ctx.binary("sub", z, b)
        main.wait_stream(side)
        return ctx.binary("add", c, s)

    side = torch.cuda.Stream()
    want = work(side).clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = work(side)
    for _ in range(20):
        got.zero_()
        graph.replay()
        assert torch.equal(got, want)
    ctx.check_device_status()


@pytest.mark.parametrize("n", [4 * 2368 * 256 - 4, 4 * 2368 * 256 + 4, 16 * 2368 * 256, 16 * 2368 * 256 + 8, 36 * 2368 * 256 + 12, 8 * 2368 * 256 + 3])
def test_elementwise_passes_of_several_items_per_thread(ctx, n):
    """Sizes at which the last pass of a grid of 2368 x 256 threads (and of any other) holds none, some or all of its items."""
    import torch

    x, y, b = torch.randn(n, device="cuda"), torch.randn(n, device="cuda"), torch.randn(4, device="cuda")
    assert torch.equal(ctx.binary("add", x, y), x + y)
    assert torch.equal(ctx.act_backprop(x, y, "relu"), torch.where(x > 0, y, torch.zeros_like(y)))
    if n % 4 == 0:
        r = x.view(n // 4, 4)
        assert torch.equal(ctx.binary("mul", r, b), r * b)
        assert torch.equal(ctx.bias_act(r, b, act="relu"), torch.relu(r + b))


@pytest.mark.parametrize("window", [(1, 3), (3, 1), (2, 3), (3, 3), (4, 2), (1, 1), (1, 2), (2, 1), (2, 2), (5, 5)])
def test_max_pool_of_quads_at_the_window_sizes_around_the_unrolled_one(ctx, oracle, window):
    x = si.uniform(91, 0, (2, 7, 6, 8), -1, 1)
    x[0, 3, 2, 1] = np.nan
    x[1, 0, 0, 2] = -np.inf
    for strides in ((1, 1), (2, 2)):
        got = host(ctx.max_pool(dev(x), window, strides, "same"))
        assert same_bits_or_both_nan(got, oracle.max_pool(x, window, strides, "same"))
