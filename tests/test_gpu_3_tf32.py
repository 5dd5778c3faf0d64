"""GPU parity of the tensor-core (tcgen05, TF32) GEMM path: matMul, 1x1 conv2d, fused epilogue.

Tolerances.  TF32 keeps 10 explicit mantissa bits of each operand, so against the exact
(double-accumulate) oracle the per-op bar is a relative Frobenius error <= 5e-3.  Against the
oracle run with the same operand rounding (products and sums still in double) only fp32
accumulation order remains, and the bar is 2e-5; whichever of truncation / round-to-nearest
matches tells how the hardware reads fp32 bits.  Small integers are exact in TF32 and every
partial sum is exact in fp32, so there the result must be bit-identical: a zero-tolerance
check of descriptors, swizzles, tile tails and the epilogue's addressing.
"""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import dev, host, plant_specials, rel_fro, same_bits, same_classes

pytestmark = pytest.mark.gpu

TF32_TOL = 5e-3
MATCHED_TOL = 2e-5

GEMM_SHAPES = [
    # M, K, N
    (128, 32, 32),        # one tile, one k-block, one MMA group
    (128, 64, 64),
    (512, 512, 512),      # config 1
    (300, 100, 72),       # ragged in M, K and N
    (1, 1024, 1000),      # batch-1 dense layer
    (128, 1024, 1000),    # batch-128 dense layer: N tail inside a 32-column chunk
    (12544, 32, 64),      # config 2 pointwise step
    (3136, 128, 128),
    (1000, 8, 16),        # K and N below one tile
    (4100, 36, 260),      # N just above one 256 tile
    (49, 1024, 1024),     # many k-blocks: the stage ring wraps several times
    (20000, 256, 512),    # more tiles than SMs: persistent loop, both accumulator stages reused
    (6272, 512, 1024),    # 196 tiles of 256 columns on 148 SMs: the 192-column tile is chosen instead
]


@pytest.mark.parametrize("mkn", GEMM_SHAPES)
def test_matmul_tf32_integer_exact(ctx, oracle, mkn):
    M, K, N = mkn
    a = si.small_integers(301, 0, (M, K), -8, 8)
    b = si.small_integers(301, 1, (K, N), -8, 8)
    got = host(ctx.matmul(dev(a), dev(b)))
    ctx.check_device_status()
    want = (a.astype(np.int64) @ b.astype(np.int64)).astype(np.float32)
    assert same_bits(got, want)


@pytest.mark.parametrize("mkn", GEMM_SHAPES)
def test_matmul_tf32_parity(ctx, oracle, mkn):
    M, K, N = mkn
    a = si.uniform(302, 0, (M, K), -1, 1)
    b = si.uniform(302, 1, (K, N), -1, 1)
    got = host(ctx.matmul(dev(a), dev(b)))
    ctx.check_device_status()
    if M * K * N <= 600_000_000:
        want = oracle.matmul(a, b)
        assert rel_fro(got, want) <= TF32_TOL
        matched = min(rel_fro(got, oracle.matmul(a, b, operand="tf32_rz")),
                      rel_fro(got, oracle.matmul(a, b, operand="tf32_rna")))
        assert matched <= MATCHED_TOL
    else:  # sampled rows, each computed one by one by the oracle
        rows = np.unique(np.linspace(0, M - 1, 257).astype(np.int64))
        want = oracle.matmul(a[rows], b)
        assert rel_fro(got[rows], want) <= TF32_TOL


SPLIT_K_SHAPES = [
    # M, K, N: few output tiles and a long K loop, so the planner cuts K into slices (work item = tile x slice)
    (128, 1024, 1000),   # dense layer at batch 128
    (1, 1024, 1000),     # dense layer at batch 1
    (49, 1024, 1024),    # pw13 at batch 1
    (196, 512, 512),     # pw7 at batch 1: two row tiles, the second mostly empty
    (300, 4100, 72),     # K not a multiple of the slice length: the last slice is short and ragged
    (512, 512, 512),     # config 1
]


@pytest.mark.parametrize("mkn", SPLIT_K_SHAPES)
def test_matmul_split_k_agrees_with_unsplit_and_oracle(ctx, oracle, monkeypatch, mkn):
    M, K, N = mkn
    a = si.uniform(311, 0, (M, K), -1, 1)
    b = si.uniform(311, 1, (K, N), -1, 1)
    monkeypatch.delenv("TFJSB_NO_SPLIT_K", raising=False)
    split = host(ctx.matmul(dev(a), dev(b)))
    again = host(ctx.matmul(dev(a), dev(b)))
    monkeypatch.setenv("TFJSB_NO_SPLIT_K", "1")
    whole = host(ctx.matmul(dev(a), dev(b)))
    ctx.check_device_status()
    assert not same_bits(split, whole)                    # another summation order: K really was cut
    assert same_bits(split, again)                        # slices are added in a fixed order, whichever finishes first
    want = oracle.matmul(a, b)
    assert rel_fro(split, want) <= TF32_TOL and rel_fro(whole, want) <= TF32_TOL
    assert rel_fro(split, oracle.matmul(a, b, operand="tf32_rz")) <= MATCHED_TOL
    ai = si.small_integers(312, 0, (M, K), -8, 8)
    bi = si.small_integers(312, 1, (K, N), -8, 8)
    monkeypatch.delenv("TFJSB_NO_SPLIT_K", raising=False)
    assert same_bits(host(ctx.matmul(dev(ai), dev(bi))), (ai.astype(np.int64) @ bi.astype(np.int64)).astype(np.float32))


def test_dense_split_k_fused_bias_and_activation(ctx, oracle):
    # the reduction applies bias and activation: [128,1,1,1024] x [1,1,1024,1000] + bias, relu6
    x = si.uniform(313, 0, (128, 1, 1, 1024), 0, 1)
    f = si.normal(313, 1, (1, 1, 1024, 1000), 0, float(np.sqrt(2.0 / 1024)))
    b = si.normal(313, 2, (1000,), 0, 0.5)
    for act in ("none", "relu6"):
        got = host(ctx.conv2d(dev(x), dev(f), bias=dev(b), act=act))
        assert rel_fro(got, oracle.conv2d(x, f, bias=b, act=act)) <= TF32_TOL
    ctx.check_device_status()


@pytest.mark.parametrize("ta,tb", [(False, True), (True, False), (True, True)])
def test_matmul_tf32_transposes(ctx, oracle, ta, tb):
    M, K, N = 260, 96, 132
    a = si.uniform(303, 0, (K, M) if ta else (M, K), -1, 1)
    b = si.uniform(303, 1, (N, K) if tb else (K, N), -1, 1)
    got = host(ctx.matmul(dev(a), dev(b), ta, tb))
    ctx.check_device_status()
    assert rel_fro(got, oracle.matmul(a, b, ta, tb)) <= TF32_TOL
    ai = si.small_integers(304, 0, a.shape, -8, 8)
    bi = si.small_integers(304, 1, b.shape, -8, 8)
    assert same_bits(host(ctx.matmul(dev(ai), dev(bi), ta, tb)), oracle.matmul(ai, bi, ta, tb))


@pytest.mark.parametrize("pair", ["0", "1"])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, False), (True, True)])
@pytest.mark.parametrize("bmkn", [(1, 4, 4, 4), (1, 36, 28, 68), (1, 132, 36, 260), (1, 260, 96, 132), (1, 300, 1000, 128), (1, 34, 520, 72),
                                  (5, 100, 36, 72), (3, 33, 64, 40)])
def test_operands_as_stored_give_the_bits_of_k_contiguous_ones(ctx, monkeypatch, bmkn, ta, tb, pair):
    """Operands stored [K, N] and [K, M] are read as they are (or transposed first, where M is no multiple of 4): the tiles'
    groups of 32 rows and atoms of 4 k end inside the matrices, the K loop is whole, in slices, or on CTA pairs.  The plan
    does not depend on the storage, so neither does any bit."""
    monkeypatch.setenv("TFJSB_GEMM_PAIR", pair)
    b, m, k, n = bmkn
    x, y = si.uniform(77, 0, (b, m, k), -1, 1), si.uniform(77, 1, (b, n, k), -1, 1)
    if b == 1:
        x, y = x[0], y[0]
    call = ctx.matmul if b == 1 else ctx.batch_matmul
    want = host(call(dev(x), dev(y), transpose_b=True))
    got = host(call(dev(np.ascontiguousarray(np.swapaxes(x, -1, -2))) if ta else dev(x), dev(y) if tb else dev(np.ascontiguousarray(np.swapaxes(y, -1, -2))),
                    transpose_a=ta, transpose_b=tb))
    ctx.check_device_status()
    assert same_bits(got, want)


def test_matmul_unaligned_shapes_take_the_cuda_core_path(ctx, oracle):
    a = si.uniform(305, 0, (70, 27), -1, 1)   # K % 4 != 0
    b = si.uniform(305, 1, (27, 33), -1, 1)   # N % 4 != 0
    got = host(ctx.matmul(dev(a), dev(b)))
    assert rel_fro(got, oracle.matmul(a, b)) <= 1e-5


@pytest.mark.parametrize("act", ["none", "relu", "relu6"])
@pytest.mark.parametrize("shape", [(1, 112, 112, 32, 64), (2, 14, 14, 512, 512), (1, 7, 7, 1024, 1024),
                                   (3, 9, 5, 8, 16), (1, 28, 28, 128, 256)])
def test_pointwise_conv_tf32_fused_epilogue(ctx, oracle, shape, act):
    N, H, W, Cin, Cout = shape
    x = si.uniform(306, 0, (N, H, W, Cin), 0, 6)
    f = si.normal(306, 1, (1, 1, Cin, Cout), 0, float(np.sqrt(2.0 / Cin)))
    b = si.normal(306, 2, (Cout,), 0, 0.5)
    got = host(ctx.conv2d(dev(x), dev(f), bias=dev(b), act=act))
    ctx.check_device_status()
    want = oracle.conv2d(x, f, bias=b, act=act)
    assert got.shape == want.shape
    assert rel_fro(got, want) <= TF32_TOL
    if act == "relu6":
        assert got.min() >= 0 and got.max() <= 6
    xi = si.small_integers(307, 0, x.shape, -8, 8)
    fi = si.small_integers(307, 1, f.shape, -8, 8)
    bi = si.small_integers(307, 2, b.shape, -8, 8)
    assert same_bits(host(ctx.conv2d(dev(xi), dev(fi), bias=dev(bi), act=act)),
                     oracle.conv2d(xi, fi, bias=bi, act=act))


IGEMM_CASES = [
    # N, H, W, Cin, fh, fw, Cout, strides, pad, dilations: conv2d as an implicit GEMM on the tensor cores
    (1, 224, 224, 3, 3, 3, 32, (2, 2), "same", (1, 1)),   # the stem of the 224 models (K = 27, scalar gather)
    (2, 33, 29, 3, 3, 3, 8, (2, 2), "same", (1, 1)),
    (1, 17, 19, 5, 3, 3, 40, (1, 1), "same", (1, 1)),     # K = 45: two k-blocks, the second mostly padding
    (1, 20, 20, 16, 3, 3, 36, (2, 2), "valid", (1, 1)),   # Cin % 4 == 0: float4 gather, K = 144
    (1, 15, 15, 4, 3, 3, 8, (1, 1), "same", (2, 2)),      # dilation
    (1, 12, 14, 7, 5, 3, 12, (3, 2), "same", (1, 1)),     # 5x3 window, unequal strides
    (3, 9, 9, 30, 1, 1, 52, (2, 2), "same", (1, 1)),      # strided 1x1
    (1, 6, 6, 72, 3, 3, 4, (1, 1), "valid", (1, 1)),      # K = 648: the stage ring wraps
    (5, 40, 40, 8, 3, 3, 260, (1, 1), "same", (1, 1)),    # Cout just above one 256-wide tile, many pixel tiles
    (3, 37, 50, 3, 3, 3, 16, (2, 2), "valid", (1, 1)),    # patch kernel: ragged tiles, 'valid'
    (2, 30, 30, 3, 3, 3, 8, (1, 1), "valid", (1, 1)),     # patch kernel: stride 1
    (1, 19, 23, 4, 2, 2, 12, (1, 1), "same", (1, 1)),     # patch kernel: 2x2 window, Cin 4, pad after only
    (2, 21, 21, 1, 5, 5, 32, (2, 2), "valid", (1, 1)),    # patch kernel: one input channel, 5x5 (K = 25)
]


@pytest.mark.parametrize("case", IGEMM_CASES)
def test_conv2d_implicit_gemm_tf32(ctx, oracle, case):
    N, H, W, Cin, fh, fw, Cout, strides, pad, dil = case
    x = si.uniform(309, 0, (N, H, W, Cin), -1, 1)
    f = si.normal(309, 1, (fh, fw, Cin, Cout), 0, float(np.sqrt(2.0 / (fh * fw * Cin))))
    b = si.normal(309, 2, (Cout,), 0, 0.5)
    got = host(ctx.conv2d(dev(x), dev(f), strides, pad, dil, dev(b), "relu6"))
    ctx.check_device_status()
    want = oracle.conv2d(x, f, strides, pad, dil, b, "relu6")
    assert got.shape == want.shape
    assert rel_fro(got, want) <= TF32_TOL
    matched = oracle.conv2d(x, f, strides, pad, dil, b, "relu6", operand="tf32_rz")
    assert rel_fro(got, matched) <= MATCHED_TOL
    xi = si.small_integers(310, 0, x.shape, -4, 4)
    fi = si.small_integers(310, 1, f.shape, -4, 4)
    assert same_bits(host(ctx.conv2d(dev(xi), dev(fi), strides, pad, dil)), oracle.conv2d(xi, fi, strides, pad, dil))
    ctx.check_device_status()


def test_separable_block_config2(ctx, oracle):
    x, layers = si.config_separable_block()
    dw, pw = layers
    y1 = ctx.depthwise_conv2d(dev(x), dev(dw.filter), dw.strides, dw.pad, dw.dilations, dev(dw.bias), dw.act)
    y2 = host(ctx.conv2d(y1, dev(pw.filter), pw.strides, pw.pad, pw.dilations, dev(pw.bias), pw.act))
    ctx.check_device_status()
    w1 = oracle.depthwise_conv2d(x, dw.filter, dw.strides, dw.pad, dw.dilations, dw.bias, dw.act)
    w2 = oracle.conv2d(w1, pw.filter, pw.strides, pw.pad, pw.dilations, pw.bias, pw.act)
    assert rel_fro(host(y1), w1) <= 1e-6
    assert rel_fro(y2, w2) <= TF32_TOL


def test_tf32_result_is_deterministic(ctx):
    a = dev(si.uniform(308, 0, (5000, 256), -1, 1))
    b = dev(si.uniform(308, 1, (256, 512), -1, 1))
    first = host(ctx.matmul(a, b))
    for _ in range(3):
        assert same_bits(host(ctx.matmul(a, b)), first)
    ctx.check_device_status()


STRIDED_CASES = [
    # batch (0: rank 2), M, K, N: rows that are no multiples of 16 bytes, fp32 accuracy on the tensor cores
    (0, 1, 1, 1),
    (0, 128, 32, 33),       # one tile and one column more
    (0, 31, 33, 129),       # the transposed tile is the smaller one
    (0, 64, 1024, 101),     # few tiles, long K: a cluster of eight
    (0, 5, 513, 7),         # a cluster, last k-block of one
    (0, 200, 150, 257),     # K % 4 != 0
    (0, 999, 66, 1001),     # more tiles than SMs
    (0, 130, 4099, 61),     # segments of the sum in each slice of K
    (7, 199, 64, 199),
    (150, 17, 19, 23),      # more products than SMs
    (3, 40, 700, 30),       # a cluster per product
]


@pytest.mark.parametrize("ta", [False, True])
@pytest.mark.parametrize("tb", [False, True])
@pytest.mark.parametrize("case", STRIDED_CASES)
def test_matmul_of_unaligned_rows(ctx, oracle, case, ta, tb):
    B, M, K, N = case
    lead = (B,) if B else ()
    sa, sb = lead + ((K, M) if ta else (M, K)), lead + ((N, K) if tb else (K, N))
    call, want = (ctx.batch_matmul, oracle.batch_matmul) if B else (ctx.matmul, oracle.matmul)
    a, b = si.small_integers(321, 0, sa, -8, 8), si.small_integers(321, 1, sb, -8, 8)
    got = host(call(dev(a), dev(b), ta, tb))  # |sums| <= 64 K < 2^24: exact in any order
    ctx.check_device_status()
    assert same_bits(got + 0.0, want(a, b, ta, tb) + 0.0)
    a, b = si.uniform(322, 0, sa, -1, 1), si.uniform(322, 1, sb, -1, 1)
    # the bar of the CUDA-core kernel
    assert rel_fro(host(call(dev(a), dev(b), ta, tb)), want(a, b, ta, tb)) <= 1e-5


@pytest.mark.parametrize("M,N,K,cuda_cores", [(131, 67, 1, True), (131, 67, 7, True), (131, 67, 16, True), (131, 67, 17, False),
                                              (19000, 9, 7, None), (9, 19001, 16, None), (19000, 101, 7, True), (27, 30001, 7, None)])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, True)])
def test_short_unaligned_products_take_the_cuda_cores(ctx, M, N, K, cuda_cores, ta, tb):
    """Where their tiles are few: one launch either way, the same bits as in fp32 mode where it is the same kernel; sums of 17
    products differ in order.  (None: as many tiles as SMs or a few more or less.)"""
    a, b = si.uniform(325, 0, (K, M) if ta else (M, K), -1, 1), si.uniform(325, 1, (N, K) if tb else (K, N), -1, 1)
    got = host(ctx.matmul(dev(a), dev(b), ta, tb))
    ctx.set_math("fp32")
    try:
        want = host(ctx.matmul(dev(a), dev(b), ta, tb))
    finally:
        ctx.set_math("tf32")
    ctx.check_device_status()
    assert cuda_cores is None or same_bits(got, want) == cuda_cores
    assert rel_fro(got, (a.T if ta else a).astype(np.float64) @ (b.T if tb else b).astype(np.float64)) <= 1.8e-8 * K ** 0.5 + 2.0 ** -24


@pytest.mark.parametrize("M,K,N,ta,tb", [(199, 64, 199, False, True), (301, 513, 303, True, True), (1301, 2001, 1303, False, False),
                                         (1301, 8191, 1303, False, True), (257, 20001, 255, True, False)])
@pytest.mark.parametrize("positive", [False, True])
def test_unaligned_products_are_as_exact_as_fp32_multiply_adds(ctx, M, K, N, ta, tb, positive):
    """Sums from 64 to 20001 products, whole and cut over clusters, of both signs and of one: the kernel that they ran on
    before, fp32 multiply-adds in order, is 1.8e-8 sqrt(K) of the result off (2^-25 per addition, errors cancelling)."""
    a, b = (si.uniform(324, i, s, 0.0 if positive else -1.0, 1.0) for i, s in ((0, (K, M) if ta else (M, K)), (1, (N, K) if tb else (K, N))))
    want = (a.T if ta else a).astype(np.float64) @ (b.T if tb else b).astype(np.float64)
    got = host(ctx.matmul(dev(a), dev(b), ta, tb))
    ctx.check_device_status()
    assert rel_fro(got, want) <= 1.8e-8 * K ** 0.5


@pytest.mark.parametrize("case", [(0, 5, 3, 7), (0, 64, 70, 101), (0, 200, 150, 257), (0, 40, 1030, 33), (7, 50, 64, 51)])
@pytest.mark.parametrize("ta,tb", [(False, False), (True, True)])
def test_unaligned_products_of_values_that_are_not_finite(ctx, case, ta, tb):
    """The same infinities and NaNs as fp32 multiply-adds give, and finite results beside them (the largest number is above
    the largest TF32 number, a NaN with low bits only below the smallest TF32 NaN)."""
    B, M, K, N = case
    lead = (B,) if B else ()
    a = si.uniform(325, 0, lead + ((K, M) if ta else (M, K)), -0.5, 0.5)
    b = si.uniform(325, 1, lead + ((N, K) if tb else (K, N)), -0.5, 0.5)
    call = ctx.batch_matmul if B else ctx.matmul
    for x, y in ((plant_specials(a, 1), b), (a, plant_specials(b, 2)), (plant_specials(a, 3), plant_specials(b, 4, largest=False)),
                 (np.full_like(a, np.inf), b), (np.full_like(a, np.nan), b)):
        got = host(call(dev(x), dev(y), ta, tb))
        ctx.set_math("fp32")
        try:
            want = host(call(dev(x), dev(y), ta, tb))
        finally:
            ctx.set_math("tf32")
        assert same_classes(got, want)
    ctx.check_device_status()


@pytest.mark.parametrize("classes", [1, 33, 101, 1001])
@pytest.mark.parametrize("batch", [1, 3, 130])
def test_unaligned_epilogue_and_dense_layer(ctx, oracle, batch, classes):
    """Bias and activation of the same kernel: a pointwise convolution and a model's dense layer."""
    from seeded_inputs.workloads import Layer

    x = si.uniform(323, 0, (batch, 5, 3, 70), -1, 1)
    f, b = si.normal(323, 1, (1, 1, 70, classes), 0, 0.2), si.normal(323, 2, (classes,), 0, 0.5)
    got = host(ctx.conv2d(dev(x), dev(f), bias=dev(b), act="relu6"))
    assert rel_fro(got, oracle.conv2d(x, f, bias=b, act="relu6")) <= 1e-5
    layer = Layer("dense", act="relu", out_channels=classes)
    layer.filter, layer.bias = si.normal(323, 3, (5 * 3 * 70, classes), 0, 0.05), b
    model = ctx.model([layer], x.shape)
    xd = dev(x)
    for graph in (False, True):
        model.set_graph(graph)
        assert rel_fro(host(model.run(xd)), oracle.run_model([layer], x)) <= 1e-5
    assert model.layer_kernels() == ["gemm_strided_kernel"]
    ctx.check_device_status()
    model.close()


IM2COL_CASES = [
    # N, H, W, Cin, fh, fw, Cout, strides, pad, dilations: A tiles fetched by im2col copies (Cin >= 16, Cin % 4 == 0)
    (1, 16, 16, 32, 3, 3, 64, (1, 1), "same", (1, 1)),
    (3, 9, 9, 16, 3, 3, 4, (1, 1), "same", (1, 1)),        # tiles run on from image to image; half-empty k-blocks
    (2, 13, 21, 64, 3, 3, 68, (1, 1), "same", (1, 1)),     # height and width differ
    (1, 1, 150, 20, 1, 3, 8, (1, 1), "same", (1, 1)),      # one row
    (2, 150, 1, 20, 3, 1, 8, (1, 1), "valid", (1, 1)),     # one column
    (2, 20, 20, 36, 3, 3, 32, (2, 2), "same", (1, 1)),     # even size: padding after only; a k-block of 4 channels
    (2, 21, 15, 48, 3, 3, 36, (2, 2), "same", (1, 1)),
    (1, 23, 19, 32, 5, 3, 12, (3, 2), "valid", (1, 1)),    # unequal window and strides, samples that nothing reads
    (1, 18, 31, 32, 3, 3, 8, (1, 1), "same", (4, 4)),      # dilation
    (2, 12, 10, 132, 2, 4, 260, (1, 1), "same", (1, 1)),   # even windows: padding after one more than before
    (4, 9, 7, 64, 1, 1, 40, (2, 2), "same", (1, 1)),       # strided 1x1
    (9, 30, 30, 64, 3, 3, 64, (1, 1), "same", (1, 1)),     # several tiles per CTA
    # a large window.  The tensor core cuts its fp32 sums at every MMA, by 7e-9 of the result on average with these operands
    # (1.8e-8 seen with others): with 33 x 33 taps, 4356 MMAs long, that alone is 3e-5; 13 x 13 taps stay below 2e-5
    (1, 40, 40, 16, 13, 13, 4, (1, 1), "valid", (1, 1)),
]


@pytest.mark.parametrize("case", IM2COL_CASES)
def test_conv2d_im2col_copies(ctx, oracle, monkeypatch, case):
    monkeypatch.setenv("TFJSB_CONV_PATCH", "0")  # which would take some of these
    N, H, W, Cin, fh, fw, Cout, strides, pad, dil = case
    K = fh * fw * Cin
    xi = si.small_integers(315, 0, (N, H, W, Cin), -4, 4)   # |sums| <= 16 K < 2^24: exact in any order
    fi = si.small_integers(315, 1, (fh, fw, Cin, Cout), -4, 4)
    got = host(ctx.conv2d(dev(xi), dev(fi), strides, pad, dil))
    ctx.check_device_status()
    assert same_bits(got, oracle.conv2d(xi, fi, strides, pad, dil))
    x = si.uniform(316, 0, xi.shape, -1, 1)
    f = si.normal(316, 1, fi.shape, 0, float(np.sqrt(2.0 / K)))
    b = si.normal(316, 2, (Cout,), 0, 0.5)
    got = host(ctx.conv2d(dev(x), dev(f), strides, pad, dil, dev(b), "relu"))
    assert rel_fro(got, oracle.conv2d(x, f, strides, pad, dil, b, "relu", operand="tf32_rz")) <= MATCHED_TOL


def test_conv2d_of_a_window_of_two_million_elements(ctx, oracle):
    """More elements than 32 rows for each block of the largest grid."""
    x, f = si.small_integers(317, 0, (1, 1025, 1026, 2), -1, 1), si.small_integers(317, 1, (1025, 1024, 2, 4), -1, 1)
    got = host(ctx.conv2d(dev(x), dev(f), (1, 1), "valid"))  # |sums| <= 2.1e6 < 2^24: exact in any order
    ctx.check_device_status()
    assert got.shape == (1, 1, 3, 4) and same_bits(got, oracle.conv2d(x, f, (1, 1), "valid"))


FUSED_BLOCK_CASES = [
    # N, H, W, C, Cout, pad: depthwise 3x3 stride 1 + pointwise, run by the executor as one fused kernel
    (1, 112, 112, 32, 64, "same"),     # config 2
    (2, 20, 37, 32, 8, "same"),        # ragged tiles in both directions, Cout below one chunk
    (3, 14, 14, 128, 128, "same"),     # four k-blocks, image smaller than the 16-wide tile
    (2, 7, 7, 256, 256, "same"),       # eight k-blocks, 256-wide accumulator (two stages)
    (1, 30, 33, 64, 100, "valid"),     # 'valid': no padding offset, Cout not a multiple of 32
    (5, 56, 56, 96, 36, "same"),       # more tiles than SMs, three k-blocks
    (2, 14, 14, 512, 512, "same"),     # two 256-wide accumulator halves sharing each A tile, 16 k-blocks
    (1, 9, 20, 64, 320, "same"),       # second half partly empty (320 = 256 + 64)
]


@pytest.mark.parametrize("case", FUSED_BLOCK_CASES)
def test_fused_depthwise_pointwise_block(ctx, oracle, monkeypatch, case):
    from seeded_inputs.workloads import Layer

    N, H, W, C, Cout, pad = case
    x = si.uniform(311, 0, (N, H, W, C), 0, 6)
    layers = [Layer("depthwise_conv2d", (3, 3), (1, 1), (1, 1), pad, "relu6", 1, "dw"),
              Layer("conv2d", (1, 1), (1, 1), (1, 1), "same", "relu6", Cout, "pw")]
    si.make_model_weights(layers, C, 311)
    model = ctx.model(layers, x.shape)
    model.set_fusion("always")                  # small cases: 'auto' would keep the layers apart
    assert model.launches_per_run == 1          # the two layers run as one kernel
    got = host(model.run(dev(x)))
    ctx.check_device_status()
    want = oracle.run_model(layers, x)
    assert got.shape == want.shape
    assert rel_fro(got, want) <= TF32_TOL
    monkeypatch.setenv("TFJSB_NO_SPLIT_K", "1")  # (a pointwise GEMM cut along K adds in another order)
    model.set_keep_all(True)                    # debug mode: the two stand-alone kernels
    unfused = host(model.run(dev(x)))
    assert model.launches_per_run == 2
    assert same_bits(got, unfused)              # same arithmetic in the same order
    monkeypatch.delenv("TFJSB_NO_SPLIT_K")
    model.close()
    # small integers: exact in TF32 and fp32, so bit-identical to the oracle
    xi = si.small_integers(312, 0, x.shape, 0, 3)
    for layer in layers:
        layer.filter = si.small_integers(312, 1, layer.filter.shape, -2, 2)
        layer.bias = si.small_integers(312, 2, layer.bias.shape, -2, 2)
        layer.act = "none"
    model = ctx.model(layers, x.shape)
    model.set_fusion("always")
    assert same_bits(host(model.run(dev(xi))), oracle.run_model(layers, xi))
    ctx.check_device_status()
    model.close()


# N, H, W, Cin, Cout, pad: 3x3, stride 1, A tiles from patches of 16 x 8 output pixels
PATCH_CASES = [
    (1, 16, 8, 32, 32, "same"),      # one whole tile, one channel block
    (1, 5, 3, 16, 4, "same"),        # smaller than a tile, half a channel block
    (2, 17, 9, 36, 68, "same"),      # one row and one column more than a tile; ragged channels
    (1, 33, 24, 64, 64, "valid"),    # no padding; the filter stays in shared memory
    (1, 20, 20, 40, 300, "same"),    # several column tiles
    (3, 14, 14, 128, 256, "same"),   # filter tiles through a ring
    (40, 9, 9, 64, 64, "same"),      # several tiles per CTA
    (2, 40, 70, 32, 96, "same"),     # an odd number of 32-column chunks per tile
]


@pytest.mark.parametrize("case", PATCH_CASES)
def test_conv2d_from_patches(ctx, oracle, monkeypatch, case):
    N, H, W, Cin, Cout, pad = case
    fh = fw = 3
    d = 1
    monkeypatch.setenv("TFJSB_CONV_PATCH", "1")
    x, f, b = si.small_integers(331, 0, (N, H, W, Cin), -3, 3), si.small_integers(331, 1, (fh, fw, Cin, Cout), -3, 3), si.small_integers(331, 2, (Cout,), -9, 9)
    for act in ("none", "relu6"):
        before = ctx.launch_count
        got = host(ctx.conv2d(dev(x), dev(f), (1, 1), pad, (d, d), bias=dev(b), act=act))
        assert ctx.launch_count == before + 1  # the other kernels for these shapes pack the filter first
        ctx.check_device_status()
        assert same_bits(got + 0.0, oracle.conv2d(x, f, (1, 1), pad, (d, d), bias=b, act=act) + 0.0)
    x, f = si.uniform(332, 0, x.shape, -1, 1), si.normal(332, 1, f.shape, 0, 0.2)
    got = host(ctx.conv2d(dev(x), dev(f), (1, 1), pad, (d, d)))
    assert rel_fro(got, oracle.conv2d(x, f, (1, 1), pad, (d, d))) <= TF32_TOL
    # operands as the tensor core reads them: fp32 sums over up to 1000 products, cut at every MMA (7e-9 of the result each)
    assert rel_fro(got, oracle.conv2d(x, f, (1, 1), pad, (d, d), operand="tf32_rz")) <= MATCHED_TOL


@pytest.mark.parametrize("case", [(1, 130, 36, 65), (1, 127, 4, 3), (1, 33, 100, 201), (3, 50, 64, 51), (5, 199, 68, 70), (3, 9, 20, 7), (1, 64, 1024, 101), (3, 50, 63, 51)])
def test_unaligned_products_with_rows_of_whole_quads(ctx, oracle, case):
    """K a multiple of 4 and N odd: K-contiguous operands are fetched four k at a time, of a batch too, whose products then
    start on 16 bytes, and the last k-block ends inside a row of tiles.  Beside them a batch whose K is no multiple of 4."""
    b, m, k, n = case
    for ta, tb in ((False, True), (False, False), (True, True)):
        x, y = si.uniform(333, 0, (b, m, k), -1, 1), si.uniform(333, 1, (b, k, n), -1, 1)
        want = np.einsum("bmk,bkn->bmn", x.astype(np.float64), y.astype(np.float64))
        xs, ys = np.ascontiguousarray(np.swapaxes(x, 1, 2)) if ta else x, np.ascontiguousarray(np.swapaxes(y, 1, 2)) if tb else y
        got = host(ctx.batch_matmul(dev(xs), dev(ys), ta, tb)) if b > 1 else host(ctx.matmul(dev(xs[0]), dev(ys[0]), ta, tb))[None]
        ctx.check_device_status()
        assert rel_fro(got, want) <= 1.8e-8 * max(k, 32) ** 0.5 + 1.2e-7  # fp32 multiply-adds, and the operands' split
