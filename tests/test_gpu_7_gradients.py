"""GPU parity of the gradient ops (conv2d / depthwiseConv2d / epilogue gradients, Sec. 3.5) against the oracle.

Bars: bit-identical on small integers (every product and partial sum exact in fp32 and in TF32, whatever the
order); fp32 CUDA-core kernels rel. Frobenius <= 1e-5; the pointwise gradients on the tensor cores <= 5e-3
against the exact oracle and <= 2e-5 against the oracle with truncated TF32 operands; the activation
gradient bit-exact.
"""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import dev, host, plant_specials, rel_fro, same_bits, same_classes

pytestmark = pytest.mark.gpu

CONV_CASES = [
    # N, H, W, Cin, Cout, fh, fw, stride, dilation, pad
    (2, 9, 11, 5, 7, 3, 3, 1, 1, "same"),
    (3, 14, 14, 8, 12, 3, 3, 2, 1, "same"),     # even size, stride 2: odd padding element after
    (2, 13, 10, 3, 32, 3, 3, 2, 1, "valid"),
    (1, 12, 12, 6, 4, 3, 3, 1, 2, "same"),      # dilated
    (2, 8, 9, 40, 36, 5, 3, 1, 1, "same"),      # more than one 32-channel tile, ragged
    (4, 31, 29, 16, 24, 3, 3, 1, 1, "same"),    # thousands of pixels: several slices in the filter gradient
    (2, 7, 5, 6, 10, 1, 1, 1, 1, "same"),       # pointwise with channel counts the tensor-core path cannot take
    (2, 9, 9, 8, 8, 1, 1, 2, 1, "same"),        # 1x1 with stride 2: not a plain matrix product
]


def geometry(oracle, H, W, fh, fw, s, d, pad):
    return oracle.window_geometry(H, fh, s, d, pad)[0], oracle.window_geometry(W, fw, s, d, pad)[0]


@pytest.mark.parametrize("case", CONV_CASES)
def test_conv2d_gradients(ctx, oracle, case):
    N, H, W, Cin, Cout, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    ctx.set_math("fp32")
    try:
        # small integers: bit-identical
        x = si.small_integers(81, 0, (N, H, W, Cin), -3, 3)
        f = si.small_integers(81, 1, (fh, fw, Cin, Cout), -3, 3)
        g = si.small_integers(81, 2, (N, Ho, Wo, Cout), -3, 3)
        dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), pad, (d, d)))
        df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), pad, (d, d)))
        ctx.check_device_status()
        assert same_bits(dx, oracle.conv2d_backprop_input(x.shape, f, g, (s, s), pad, (d, d)))
        assert same_bits(df, oracle.conv2d_backprop_filter(x, f.shape, g, (s, s), pad, (d, d)))
        # random values
        x = si.uniform(82, 0, (N, H, W, Cin), -1, 1)
        f = si.normal(82, 1, (fh, fw, Cin, Cout), 0, 0.3)
        g = si.normal(82, 2, (N, Ho, Wo, Cout), 0, 1)
        dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), pad, (d, d)))
        df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), pad, (d, d)))
        ctx.check_device_status()
        assert rel_fro(dx, oracle.conv2d_backprop_input(x.shape, f, g, (s, s), pad, (d, d))) <= 1e-5
        assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g, (s, s), pad, (d, d))) <= 1e-5
    finally:
        ctx.set_math("tf32")


@pytest.mark.parametrize("case", CONV_CASES[:6])
@pytest.mark.parametrize("mult", [1, 2])
def test_depthwise_gradients(ctx, oracle, case, mult):
    N, H, W, C, _, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    x = si.small_integers(83, 0, (N, H, W, C), -3, 3)
    f = si.small_integers(83, 1, (fh, fw, C, mult), -3, 3)
    g = si.small_integers(83, 2, (N, Ho, Wo, C * mult), -3, 3)
    dx = host(ctx.depthwise_conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), pad, (d, d)))
    df = host(ctx.depthwise_conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), pad, (d, d)))
    ctx.check_device_status()
    assert same_bits(dx, oracle.depthwise_conv2d_backprop_input(x.shape, f, g, (s, s), pad, (d, d)))
    assert same_bits(df, oracle.depthwise_conv2d_backprop_filter(x, f.shape, g, (s, s), pad, (d, d)))
    x = si.uniform(84, 0, (N, H, W, C), -1, 1)
    f = si.normal(84, 1, (fh, fw, C, mult), 0, 0.5)
    g = si.normal(84, 2, (N, Ho, Wo, C * mult), 0, 1)
    dx = host(ctx.depthwise_conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), pad, (d, d)))
    df = host(ctx.depthwise_conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), pad, (d, d)))
    ctx.check_device_status()
    assert rel_fro(dx, oracle.depthwise_conv2d_backprop_input(x.shape, f, g, (s, s), pad, (d, d))) <= 1e-6
    assert rel_fro(df, oracle.depthwise_conv2d_backprop_filter(x, f.shape, g, (s, s), pad, (d, d))) <= 1e-5


SPLIT_CASES = [
    # N, H, W, Cin, Cout, fh, fw, stride, dilation, pad: fp32 gradients on the tensor cores in TF32 mode
    (1, 5, 5, 4, 4, 3, 3, 1, 1, "same"),         # everything smaller than a tile
    (2, 16, 16, 32, 32, 3, 3, 1, 1, "same"),
    (3, 13, 17, 36, 68, 3, 3, 1, 1, "same"),     # ragged channel blocks, two 64-wide column tiles or one of 128
    (2, 12, 12, 160, 40, 3, 3, 1, 1, "valid"),   # five 32-channel blocks: M tiles across taps
    (2, 14, 15, 40, 132, 3, 3, 2, 1, "same"),    # four residue classes, two column tiles of dy
    (2, 15, 14, 24, 20, 3, 3, 2, 1, "valid"),    # samples that no output reads
    (1, 17, 19, 16, 16, 5, 4, 3, 1, "same"),     # nine classes, uneven numbers of taps
    (2, 11, 13, 16, 8, 2, 2, 4, 1, "same"),      # classes without a tap: exact zeros
    (2, 9, 9, 8, 8, 1, 1, 2, 1, "same"),         # strided 1x1
    (1, 14, 18, 32, 24, 3, 3, 1, 2, "same"),     # dilated
    (2, 8, 9, 3, 32, 3, 3, 2, 1, "same"),        # three input channels: input gradient with scalar stores
    (2, 9, 11, 6, 12, 1, 1, 1, 1, "same"),       # pointwise, Cin no multiple of 4
    (1, 7, 7, 128, 256, 3, 3, 1, 1, "same"),     # few tiles, long K: parts of the K loop
    (24, 28, 28, 64, 64, 3, 3, 1, 1, "same"),    # several tiles per CTA, slices of 32 pixel blocks
]


@pytest.mark.parametrize("case", SPLIT_CASES)
def test_conv2d_gradients_keep_fp32_accuracy_in_tf32_mode(ctx, oracle, case):
    N, H, W, Cin, Cout, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    args = ((s, s), pad, (d, d))
    # small integers: hi parts and their products exact, lo parts zero
    x = si.small_integers(93, 0, (N, H, W, Cin), -3, 3)
    f = si.small_integers(93, 1, (fh, fw, Cin, Cout), -3, 3)
    g = si.small_integers(93, 2, (N, Ho, Wo, Cout), -3, 3)
    dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), *args))
    df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), *args))
    ctx.check_device_status()
    assert same_bits(dx + 0.0, oracle.conv2d_backprop_input(x.shape, f, g, *args) + 0.0)
    assert same_bits(df + 0.0, oracle.conv2d_backprop_filter(x, f.shape, g, *args) + 0.0)
    # the bar of the CUDA-core kernels; long sums and a tighter bar: test_conv2d_gradients_are_as_exact_as_fp32_multiply_adds
    x = si.uniform(94, 0, x.shape, -1, 1)
    f = si.normal(94, 1, f.shape, 0, 0.3)
    g = si.normal(94, 2, g.shape, 0, 1)
    dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), *args))
    df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), *args))
    ctx.check_device_status()
    assert rel_fro(dx, oracle.conv2d_backprop_input(x.shape, f, g, *args)) <= 1e-5
    # a pointwise filter gradient with a multiple of 4 pixels is a TF32 product
    assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g, *args)) <= 1e-5


@pytest.fixture
def tensor_core_input_gradient(monkeypatch):
    """Short sums run on the CUDA cores by default: the tensor-core kernel wherever it can, for its small cases."""
    monkeypatch.setenv("TFJSB_GRAD_INPUT", "1")


@pytest.mark.parametrize("case", SPLIT_CASES)
def test_both_input_gradients_of_short_sums(ctx, oracle, case, tensor_core_input_gradient, monkeypatch):
    N, H, W, Cin, Cout, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    f, g = si.small_integers(93, 1, (fh, fw, Cin, Cout), -3, 3), si.small_integers(93, 2, (N, Ho, Wo, Cout), -3, 3)
    want = oracle.conv2d_backprop_input((N, H, W, Cin), f, g, (s, s), pad, (d, d)) + 0.0
    for cores in ("1", "0"):
        monkeypatch.setenv("TFJSB_GRAD_INPUT", cores)
        assert same_bits(host(ctx.conv2d_backprop_input((N, H, W, Cin), dev(f), dev(g), (s, s), pad, (d, d))) + 0.0, want)
    monkeypatch.setenv("TFJSB_GRAD_INPUT", "1")
    f, g = si.normal(94, 1, f.shape, 0, 0.3), si.normal(94, 2, g.shape, 0, 1)
    dx = host(ctx.conv2d_backprop_input((N, H, W, Cin), dev(f), dev(g), (s, s), pad, (d, d)))
    ctx.check_device_status()
    assert rel_fro(dx, oracle.conv2d_backprop_input((N, H, W, Cin), f, g, (s, s), pad, (d, d))) <= 1e-5


@pytest.mark.parametrize("case", [(2, 14, 14, 16, 32, 3, 3, 1), (24, 28, 28, 64, 64, 3, 3, 1), (4, 14, 14, 512, 512, 3, 3, 1), (1, 20, 20, 256, 512, 5, 5, 1),
                                  (2, 56, 56, 32, 64, 3, 3, 2)])
def test_conv2d_gradients_are_as_exact_as_fp32_multiply_adds(ctx, oracle, case):
    """Long sums too: the input gradient's are over taps and output channels, 288 to 12800 products, the filter gradient's
    over pixels, of which a partial sum takes 1024 at least.  fp32 multiply-adds in order, the kernels before, are
    1.8e-8 sqrt(K) off (2^-25 per addition, errors cancelling); the oracle's result is rounded to fp32 (2.5e-8)."""
    N, H, W, Cin, Cout, fh, fw, s = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, 1, "same")
    x = si.uniform(97, 0, (N, H, W, Cin), 0, 6)
    f = si.normal(97, 1, (fh, fw, Cin, Cout), 0, float(np.sqrt(2.0 / (fh * fw * Cin))))
    g = si.normal(97, 2, (N, Ho, Wo, Cout), 0, 1)
    dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), "same"))
    df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), "same"))
    ctx.check_device_status()
    products = fh * fw * Cout / (s * s)  # of the average residue class
    assert rel_fro(dx, oracle.conv2d_backprop_input(x.shape, f, g, (s, s), "same")) <= 1.8e-8 * products ** 0.5 + 2.5e-8
    assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g, (s, s), "same")) <= 1.8e-8 * min(N * Ho * Wo, 1024) ** 0.5 + 2.5e-8


@pytest.mark.parametrize("case", [SPLIT_CASES[i] for i in (0, 2, 4, 5, 7, 9, 11, 12)])
@pytest.mark.parametrize("planted", ["x", "f", "g", "all"])
def test_conv2d_gradients_of_values_that_are_not_finite(ctx, oracle, case, planted, tensor_core_input_gradient):
    """The same infinities and NaNs as the CUDA-core kernels give, also at the border, where the copied tiles hold zeros for
    what does not exist: an infinite filter value reaches no sample through a tap that it does not meet."""
    N, H, W, Cin, Cout, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    args = ((s, s), pad, (d, d))
    x, f, g = si.uniform(98, 0, (N, H, W, Cin), -1, 1), si.normal(98, 1, (fh, fw, Cin, Cout), 0, 0.2), si.normal(98, 2, (N, Ho, Wo, Cout), 0, 0.5)
    if planted in ("x", "all"):
        x = plant_specials(x, 5, (0, x.size - 1), planted != "all")
    if planted in ("f", "all"):
        f = plant_specials(f, 6, (0, f.size - 1), planted != "all")
    if planted in ("g", "all"):
        g = plant_specials(g, 7, (0, g.size - 1), planted != "all")

    def both():
        return (host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g), *args)), host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g), *args)))

    got = both()
    ctx.check_device_status()
    ctx.set_math("fp32")
    try:
        want = both()
    finally:
        ctx.set_math("tf32")
    assert same_classes(got[0], want[0]) and same_classes(got[1], want[1])


SMALL_FILTER_CASES = [
    # N, H, W, Cin, Cout, fh, fw, stride, dilation, pad: windows of up to 32 elements
    (1, 3, 3, 3, 4, 3, 3, 1, 1, "same"),
    (2, 31, 17, 3, 32, 3, 3, 2, 1, "same"),      # four pixel lanes per channel group
    (3, 40, 33, 3, 64, 3, 3, 1, 1, "same"),      # two
    (2, 29, 30, 3, 100, 3, 3, 2, 1, "valid"),    # one, ragged channels
    (2, 20, 21, 3, 260, 3, 3, 1, 1, "same"),     # three channel tiles
    (1, 1, 90, 1, 36, 1, 5, 1, 1, "same"),       # one row
    (70, 9, 5, 2, 8, 4, 4, 1, 1, "same"),        # 32 elements; images smaller than a step of pixels
    (2, 24, 18, 3, 16, 3, 3, 1, 3, "same"),      # dilated
]


@pytest.mark.parametrize("math", ["tf32", "fp32"])
@pytest.mark.parametrize("case", SMALL_FILTER_CASES)
def test_gradient_of_a_small_filter(ctx, oracle, case, math):
    N, H, W, Cin, Cout, fh, fw, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, fh, fw, s, d, pad)
    ctx.set_math(math)
    try:
        x = si.small_integers(95, 0, (N, H, W, Cin), -3, 3)
        g = si.small_integers(95, 1, (N, Ho, Wo, Cout), -3, 3)
        df = host(ctx.conv2d_backprop_filter(dev(x), (fh, fw, Cin, Cout), dev(g), (s, s), pad, (d, d)))
        assert same_bits(df + 0.0, oracle.conv2d_backprop_filter(x, (fh, fw, Cin, Cout), g, (s, s), pad, (d, d)) + 0.0)
        x, g = si.uniform(96, 0, x.shape, -1, 1), si.normal(96, 1, g.shape, 0, 1)
        df = host(ctx.conv2d_backprop_filter(dev(x), (fh, fw, Cin, Cout), dev(g), (s, s), pad, (d, d)))
        assert rel_fro(df, oracle.conv2d_backprop_filter(x, (fh, fw, Cin, Cout), g, (s, s), pad, (d, d))) <= 1e-5
    finally:
        ctx.set_math("tf32")
    ctx.check_device_status()


DEPTHWISE_3X3_CASES = [
    # N, H, W, C, stride, dilation, pad: tile edges of the pipelined kernels and of the stride-2 column pairs
    (1, 1, 1, 4, 1, 1, "same"),
    (2, 7, 7, 100, 1, 1, "same"),      # 8-wide tiles, a ragged channel block
    (3, 14, 17, 64, 1, 1, "same"),     # one column past a 16-wide tile
    (2, 9, 33, 36, 1, 1, "valid"),     # mirrored padding of two
    (1, 13, 20, 8, 1, 2, "same"),      # dilated: register kernel forward over dy, per-tap filter gradient
    (2, 20, 18, 32, 1, 4, "same"),
    (2, 1, 2, 4, 2, 1, "same"),
    (2, 16, 16, 32, 2, 1, "same"),     # even size: padding after only
    (3, 15, 31, 40, 2, 1, "same"),     # odd size: padding on both sides
    (2, 18, 35, 68, 2, 1, "valid"),    # an input row that no output reads
    (70, 28, 28, 128, 1, 1, "same"),   # several tiles per CTA
    (70, 28, 29, 96, 2, 1, "same"),
]


@pytest.mark.parametrize("case", DEPTHWISE_3X3_CASES)
def test_depthwise_3x3_gradients_at_tile_edges(ctx, oracle, case):
    N, H, W, C, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, 3, 3, s, d, pad)
    # small integers: |df| <= 9 * N * Ho * Wo < 2^24, exact in any order
    x = si.small_integers(91, 0, (N, H, W, C), -3, 3)
    f = si.small_integers(91, 1, (3, 3, C, 1), -3, 3)
    g = si.small_integers(91, 2, (N, Ho, Wo, C), -3, 3)
    dx = host(ctx.depthwise_conv2d_backprop_input(x.shape, dev(f), dev(g), (s, s), pad, (d, d)))
    df = host(ctx.depthwise_conv2d_backprop_filter(dev(x), f.shape, dev(g), (s, s), pad, (d, d)))
    ctx.check_device_status()
    assert same_bits(dx + 0.0, oracle.depthwise_conv2d_backprop_input(x.shape, f, g, (s, s), pad, (d, d)) + 0.0)
    assert same_bits(df + 0.0, oracle.depthwise_conv2d_backprop_filter(x, f.shape, g, (s, s), pad, (d, d)) + 0.0)


@pytest.mark.parametrize("case", [DEPTHWISE_3X3_CASES[i] for i in (0, 1, 2, 3, 4, 5, 7, 8, 9, 10)])
@pytest.mark.parametrize("planted", ["x", "f", "g", "all"])
def test_depthwise_3x3_gradients_of_values_that_are_not_finite(ctx, oracle, case, planted):
    """A sample that does not exist takes part in no sum: an infinite dy at the border, or an infinite filter value, makes no
    NaN of it."""
    N, H, W, C, s, d, pad = case
    Ho, Wo = geometry(oracle, H, W, 3, 3, s, d, pad)
    args = ((s, s), pad, (d, d))
    x, f, g = si.uniform(99, 0, (N, H, W, C), -1, 1), si.normal(99, 1, (3, 3, C, 1), 0, 0.3), si.normal(99, 2, (N, Ho, Wo, C), 0, 0.5)
    if planted in ("x", "all"):
        x = plant_specials(x, 5, (0, x.size - 1), planted != "all")
    if planted in ("f", "all"):
        f = plant_specials(f, 6, (0, f.size - 1), planted != "all")
    if planted in ("g", "all"):
        g = plant_specials(g, 7, (0, g.size - 1), planted != "all")
    dx = host(ctx.depthwise_conv2d_backprop_input(x.shape, dev(f), dev(g), *args))
    df = host(ctx.depthwise_conv2d_backprop_filter(dev(x), f.shape, dev(g), *args))
    ctx.check_device_status()
    assert same_classes(dx, oracle.depthwise_conv2d_backprop_input(x.shape, f, g, *args))
    assert same_classes(df, oracle.depthwise_conv2d_backprop_filter(x, f.shape, g, *args))


@pytest.mark.parametrize("shape", [(1, 1), (1024, 3), (1025, 32), (5000, 101), (3000, 8192), (40, 3, 7, 4), (1 << 17, 4), (70001, 36)])
def test_bias_gradient_slices(ctx, oracle, shape):
    dz = si.small_integers(92, 0, shape, -8, 8)  # |sums| <= 8 * 2^17: exact in any order
    assert same_bits(host(ctx.bias_backprop(dev(dz))), oracle.bias_backprop(dz))


POINTWISE_CASES = [
    # N, H, W, Cin, Cout: gradients of a 1x1 convolution as matrix products on the tensor cores
    (1, 8, 8, 32, 64),        # 64 pixels: a single slice, K = 64
    (2, 28, 28, 128, 256),    # pw4 of the 224 model at batch 2: 1568 pixels
    (8, 56, 56, 64, 128),     # pw2 at batch 8: 25088 pixels cut into slices, batched launch + ordered sum
    (3, 15, 15, 36, 20),      # 675 pixels: not a multiple of 4, so the filter gradient falls back to CUDA cores
    (2, 14, 14, 512, 512),    # pw7-pw11
]


@pytest.mark.parametrize("case", POINTWISE_CASES)
def test_pointwise_gradients_on_the_tensor_cores(ctx, oracle, case):
    N, H, W, Cin, Cout = case
    before = ctx.launch_count
    x = si.small_integers(85, 0, (N, H, W, Cin), -2, 2)
    f = si.small_integers(85, 1, (1, 1, Cin, Cout), -2, 2)
    g = si.small_integers(85, 2, (N, H, W, Cout), -2, 2)
    dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g)))
    df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g)))
    ctx.check_device_status()
    assert ctx.launch_count > before
    # |sums| <= 4 * max(Cout, N*H*W) < 2^24: exact whatever the order and the multiplier
    assert same_bits(dx, oracle.conv2d_backprop_input(x.shape, f, g))
    assert same_bits(df, oracle.conv2d_backprop_filter(x, f.shape, g))
    x = si.uniform(86, 0, (N, H, W, Cin), -1, 1)
    f = si.normal(86, 1, (1, 1, Cin, Cout), 0, 0.3)
    g = si.normal(86, 2, (N, H, W, Cout), 0, 1)
    dx = host(ctx.conv2d_backprop_input(x.shape, dev(f), dev(g)))
    df = host(ctx.conv2d_backprop_filter(dev(x), f.shape, dev(g)))
    ctx.check_device_status()
    assert rel_fro(dx, oracle.conv2d_backprop_input(x.shape, f, g)) <= 5e-3
    assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g)) <= 5e-3
    # against the oracle whose operands are truncated the way the tensor core reads them
    assert rel_fro(dx, oracle.conv2d_backprop_input(x.shape, f, g, operand="tf32_rz")) <= 2e-5
    if (N * H * W) % 4 == 0:
        assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g, operand="tf32_rz")) <= 2e-5
    else:
        assert rel_fro(df, oracle.conv2d_backprop_filter(x, f.shape, g)) <= 1e-5


def test_epilogue_gradients(ctx, oracle):
    y = np.array([-0.0, 0.0, 1e-30, 0.5, 5.999999, 6.0, 3.0, 0.0], np.float32)
    dy = np.array([1, 2, 3, 4, 5, 6, -7, np.nan], np.float32)
    for act in ("none", "relu", "relu6"):
        assert same_bits(host(ctx.act_backprop(dev(y), dev(dy), act)), oracle.act_backprop(y, dy, act)), act
    z = si.uniform(87, 0, (5, 17, 13, 24), -3, 9)
    g = si.normal(87, 1, z.shape, 0, 1)
    for act in ("relu", "relu6"):
        yv = oracle.bias_act(z, None, act)
        assert same_bits(host(ctx.act_backprop(dev(yv), dev(g), act)), oracle.act_backprop(yv, g, act)), act
    # bias gradient: exact on integers (one slice and many), 1e-6 otherwise
    for shape in [(3, 4, 5, 6), (64, 28, 28, 40), (7, 1000)]:
        dz = si.small_integers(88, 0, shape, -8, 8)
        assert same_bits(host(ctx.bias_backprop(dev(dz))), oracle.bias_backprop(dz)), shape
        dz = si.normal(88, 1, shape, 0, 1)
        want = oracle.bias_backprop(dz)
        assert np.max(np.abs(host(ctx.bias_backprop(dev(dz))) - want)) <= 1e-5 * np.sqrt(dz.size / shape[-1]), shape
    ctx.check_device_status()


def test_gradients_reject_bad_arguments(ctx, tfjsb):
    import torch

    f = torch.zeros(3, 3, 4, 8, device="cuda")
    with pytest.raises(tfjsb.TfjsbError) as e:  # dy does not have the forward output's shape
        ctx.conv2d_backprop_input((1, 8, 8, 4), f, torch.zeros(1, 8, 8, 6, device="cuda"))
    assert e.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as e:  # filter channels differ from x's
        ctx.conv2d_backprop_filter(torch.zeros(1, 8, 8, 5, device="cuda"), (3, 3, 4, 8), torch.zeros(1, 8, 8, 8, device="cuda"))
    assert e.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as e:
        ctx.depthwise_conv2d_backprop_input((1, 8, 8, 4), torch.zeros(3, 3, 4, 1, device="cuda"),
                                            torch.zeros(1, 4, 4, 4, device="cuda"), (2, 2), "same", (2, 2))
    assert e.value.status_name == "UNSUPPORTED"
    with pytest.raises(tfjsb.TfjsbError) as e:
        ctx.bias_backprop(torch.zeros(4, 6, device="cuda"), out=torch.zeros(5, device="cuda"))
    assert e.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as e:
        ctx.act_backprop(torch.zeros(4, 6, device="cuda"), torch.zeros(4, 7, device="cuda"), "relu")
    assert e.value.status_name == "SHAPE"
    # scratch sized up front: a later call finds it large enough and allocates nothing
    ctx.reserve_scratch(8 << 20)
    x = torch.ones(2, 16, 16, 32, device="cuda")
    out = torch.empty(1, 1, 32, 64, device="cuda")
    dy = torch.ones(2, 16, 16, 64, device="cuda")
    ctx.conv2d_backprop_filter(x, (1, 1, 32, 64), dy, out=out)  # first use loads the kernels' code
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ctx.conv2d_backprop_filter(x, (1, 1, 32, 64), dy, out=out.zero_())
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == free0
    assert torch.equal(out, torch.full_like(out, 512.0))


def test_gradients_in_a_capture_without_scratch(tfjsb, oracle):
    """A context that has allocated nothing yet, first used inside a stream capture, where it must not allocate: the gradients
    do without partial results, and a convolution whose reserved scratch holds the plainly packed filter only uses that."""
    import torch

    own = tfjsb.Context(0)
    own.reserve_scratch(5120)  # 8 output channels x 160 (3 x 3 x 16 window elements, padded to whole k-blocks) x 4 bytes
    x, f, g = si.small_integers(101, 0, (1, 7, 7, 128), -3, 3), si.small_integers(101, 1, (3, 3, 128, 256), -3, 3), si.small_integers(101, 2, (1, 7, 7, 256), -3, 3)
    fd, gd = si.small_integers(101, 3, (3, 3, 128, 1), -3, 3), si.small_integers(101, 4, (1, 7, 7, 128), -3, 3)
    x3, g3 = si.small_integers(101, 5, (2, 20, 20, 3), -3, 3), si.small_integers(101, 6, (2, 20, 20, 32), -3, 3)
    x16, f16 = si.small_integers(101, 7, (1, 9, 9, 16), -3, 3), si.small_integers(101, 8, (3, 3, 16, 8), -3, 3)
    rows = si.small_integers(101, 9, (5000, 40), -8, 8)
    d = {k: dev(v) for k, v in dict(x=x, f=f, g=g, fd=fd, gd=gd, x3=x3, g3=g3, x16=x16, f16=f16, rows=rows).items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = [own.conv2d_backprop_input(x.shape, d["f"], d["g"]), own.conv2d_backprop_filter(d["x"], f.shape, d["g"]),
               own.conv2d_backprop_filter(d["x3"], (3, 3, 3, 32), d["g3"]), own.depthwise_conv2d_backprop_filter(d["x"], fd.shape, d["gd"]),
               own.bias_backprop(d["rows"]), own.conv2d(d["x16"], d["f16"])]
    graph.replay()
    torch.cuda.synchronize()
    want = [oracle.conv2d_backprop_input(x.shape, f, g), oracle.conv2d_backprop_filter(x, f.shape, g),
            oracle.conv2d_backprop_filter(x3, (3, 3, 3, 32), g3), oracle.depthwise_conv2d_backprop_filter(x, fd.shape, gd),
            oracle.bias_backprop(rows), oracle.conv2d(x16, f16)]
    own.check_device_status()
    for a, b in zip(got, want):
        assert same_bits(host(a) + 0.0, b + 0.0)
    del graph, got
    own.close()


@pytest.mark.parametrize("case", [(1, 16, 8, 32, 32, "same"), (1, 5, 3, 4, 16, "same"), (2, 17, 9, 36, 68, "same"), (1, 33, 24, 64, 64, "valid"),
                                  (1, 20, 20, 300, 40, "same"), (2, 14, 14, 128, 512, "same"), (30, 9, 20, 64, 32, "same")])
def test_conv2d_input_gradient_from_patches(ctx, oracle, monkeypatch, case):
    """Stride 1, tiles of 16 x 8 samples: taps last to first, the forward padding's complement, parts of the K loop."""
    N, H, W, Cin, Cout, pad = case
    fh, fw, d = 3, 3, 1
    monkeypatch.setenv("TFJSB_CONV_PATCH", "1")
    Ho, Wo = geometry(oracle, H, W, fh, fw, 1, d, pad)
    shape, args = (N, H, W, Cin), ((1, 1), pad, (d, d))
    f, g = si.small_integers(99, 1, (fh, fw, Cin, Cout), -3, 3), si.small_integers(99, 2, (N, Ho, Wo, Cout), -3, 3)
    got = host(ctx.conv2d_backprop_input(shape, dev(f), dev(g), *args))
    ctx.check_device_status()
    assert same_bits(got + 0.0, oracle.conv2d_backprop_input(shape, f, g, *args) + 0.0)
    f, g = si.normal(99, 3, f.shape, 0, 0.2), si.normal(99, 4, g.shape, 0, 1)
    got = host(ctx.conv2d_backprop_input(shape, dev(f), dev(g), *args))
    if Cout > 32:  # sums over channels first and taps second, not the other way round: other bits than the other kernel's
        with monkeypatch.context() as m:
            m.setenv("TFJSB_CONV_PATCH", "0")
            m.setenv("TFJSB_GRAD_INPUT", "1")
            assert not same_bits(got, host(ctx.conv2d_backprop_input(shape, dev(f), dev(g), *args)))
    # fp32 multiply-adds in order, 1.8e-8 sqrt(K), the operands' split, the oracle's rounding
    assert rel_fro(got, oracle.conv2d_backprop_input(shape, f, g, *args)) <= 1.8e-8 * (fh * fw * Cout) ** 0.5 + 1.2e-7
    # infinities and NaNs as fp32 multiply-adds give them, at the border too
    f, g = plant_specials(f, 6, (0, f.size - 1), False), plant_specials(g, 7, (0, g.size - 1), False)
    got = host(ctx.conv2d_backprop_input(shape, dev(f), dev(g), *args))
    ctx.set_math("fp32")
    try:
        want = host(ctx.conv2d_backprop_input(shape, dev(f), dev(g), *args))
    finally:
        ctx.set_math("tf32")
    assert same_classes(got, want)


def test_the_input_gradient_switch_decides_where_patches_would_run(ctx, monkeypatch):
    """Sums of the three kernels differ in order, so in the last bits: 0 is the kernel of the fp32 mode, 1 the one that runs
    without patches, unset the patches, which the same shape takes by rule."""
    shape, f, g = (4, 14, 14, 512), dev(si.normal(101, 1, (3, 3, 512, 512), 0, 0.2)), dev(si.normal(101, 2, (4, 14, 14, 512), 0, 1))
    monkeypatch.setenv("TFJSB_CONV_PATCH", "1")
    patches = host(ctx.conv2d_backprop_input(shape, f, g))
    monkeypatch.setenv("TFJSB_CONV_PATCH", "0")
    monkeypatch.setenv("TFJSB_GRAD_INPUT", "1")
    any_window = host(ctx.conv2d_backprop_input(shape, f, g))
    monkeypatch.delenv("TFJSB_CONV_PATCH")
    ctx.set_math("fp32")
    try:
        cuda_cores = host(ctx.conv2d_backprop_input(shape, f, g))
    finally:
        ctx.set_math("tf32")
    assert not same_bits(patches, any_window) and not same_bits(patches, cuda_cores) and not same_bits(any_window, cuda_cores)
    assert same_bits(host(ctx.conv2d_backprop_input(shape, f, g)), any_window)
    monkeypatch.setenv("TFJSB_GRAD_INPUT", "0")
    assert same_bits(host(ctx.conv2d_backprop_input(shape, f, g)), cuda_cores)
    monkeypatch.delenv("TFJSB_GRAD_INPUT")
    assert same_bits(host(ctx.conv2d_backprop_input(shape, f, g)), patches)
    ctx.check_device_status()


@pytest.mark.parametrize("case,forward,gradient", [((63, 28, 28, 128, 256), False, None), ((2, 56, 56, 64, 64), True, None), ((61, 28, 28, 128, 120), None, False),
                                                   ((42, 7, 7, 128, 128), None, False), ((9, 8, 8, 512, 112), None, True)])
def test_which_3x3_convolutions_run_from_patches(ctx, monkeypatch, case, forward, gradient):
    """By estimate.  Images that 16 x 8 pixels divide badly took up to 1.7 times as long from patches; the bits, sums in
    another order, show which kernel ran."""
    import torch

    N, H, W, Cin, Cout = case
    gen = torch.Generator(device="cuda").manual_seed(5)
    x, f, g = (torch.randn(shape, generator=gen, device="cuda") for shape in ((N, H, W, Cin), (3, 3, Cin, Cout), (N, H, W, Cout)))
    for call, taken in ((lambda: ctx.conv2d(x, f), forward), (lambda: ctx.conv2d_backprop_input(x.shape, f, g), gradient)):
        if taken is None:
            continue
        monkeypatch.delenv("TFJSB_CONV_PATCH", raising=False)
        chosen = call()
        monkeypatch.setenv("TFJSB_CONV_PATCH", "1")
        patches = call()
        monkeypatch.setenv("TFJSB_CONV_PATCH", "0")
        copies = call()
        assert not torch.equal(patches, copies)
        assert torch.equal(chosen, patches if taken else copies)
    ctx.check_device_status()


@pytest.mark.parametrize("patches", ["0", "1"])
def test_long_sums_of_both_input_gradient_kernels(ctx, oracle, monkeypatch, patches):
    """4608 products: the bound of fp32 multiply-adds in order, as for the other shapes above."""
    monkeypatch.setenv("TFJSB_CONV_PATCH", patches)
    f, g = si.normal(97, 1, (3, 3, 512, 512), 0, float(np.sqrt(2.0 / 4608))), si.normal(97, 2, (4, 14, 14, 512), 0, 1)
    got = host(ctx.conv2d_backprop_input((4, 14, 14, 512), dev(f), dev(g), (1, 1), "same"))
    ctx.check_device_status()
    assert rel_fro(got, oracle.conv2d_backprop_input((4, 14, 14, 512), f, g, (1, 1), "same")) <= 1.8e-8 * 4608 ** 0.5 + 2.5e-8
