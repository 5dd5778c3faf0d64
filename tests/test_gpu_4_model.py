"""GPU parity of the graph executor on the MobileNet-v1-style configs.

Whole-model bar: max |logit_gpu - logit_oracle| <= 1e-2 * (max logit - min logit) per image, and
the same top-1 class.  With random weights two logits can nearly tie, so each image's oracle
top-1 / top-2 margin is checked first: it must be at least 4x the tolerance, otherwise the
top-1 comparison would be testing luck (if a seed ever fails this, change the seed and say so).
"""
import numpy as np
import pytest

import seeded_inputs as si
from helpers import dev, host, rel_fro, same_bits

pytestmark = pytest.mark.gpu


def logits_and_probs(model, x_dev):
    probs = model.run(x_dev)
    logits = model.layer_output(model.n_layers - 2)
    return host(logits), host(probs)


def check_against_oracle(got_logits, got_probs, want_logits, want_probs, rel=1e-2):
    for i in range(want_logits.shape[0]):
        span = float(want_logits[i].max() - want_logits[i].min())
        tol = rel * span
        top = np.sort(want_logits[i])
        err = float(np.max(np.abs(got_logits[i] - want_logits[i])))
        assert err <= tol, f"image {i}: max logit error {err:.3e} > {tol:.3e}"
        if rel >= 1e-2:
            assert top[-1] - top[-2] >= 4 * tol, f"image {i}: oracle top-1 margin too small; pick another seed"
        assert int(got_logits[i].argmax()) == int(want_logits[i].argmax())
        assert int(got_probs[i].argmax()) == int(want_probs[i].argmax())
        assert abs(float(got_probs[i].astype(np.float64).sum()) - 1) <= 1e-5
    return True


@pytest.mark.parametrize("math", ["tf32", "fp32"])
def test_small_model_every_layer(ctx, oracle, math):
    """A reduced model (alpha 0.25, 64x64 input, batch 3): every layer's output against the oracle."""
    x, layers = si.config_mobilenet(0.25, 64, 3, seed=4243, classes=100)
    want = oracle.run_model(layers, x, keep_all=True)
    ctx.set_math(math)
    try:
        model = ctx.model(layers, x.shape)
    finally:
        ctx.set_math("tf32")
    model.set_keep_all(True)
    probs = host(model.run(dev(x)))
    ctx.check_device_status()
    assert model.launches_per_run == len(layers) == 30  # keep-all mode runs every layer on its own
    tol = 2e-2 if math == "tf32" else 1e-4  # per-layer drift accumulates through 27 conv layers
    # Each layer on its own, at the per-op bar: the oracle applied to the input the GPU layer actually read
    # (the GPU's previous output), so that no drift from earlier layers is in the comparison.
    op_tol = 5e-3 if math == "tf32" else 1e-5
    prev = x
    for i, layer in enumerate(layers):
        got = host(model.layer_output(i)) if i < len(layers) - 1 else probs
        assert got.shape == want[i].shape, layer.name
        assert rel_fro(got, want[i]) <= tol, f"layer {i} ({layer.name}) diverges: {rel_fro(got, want[i]):.3e}"
        alone = oracle.run_model([layer], prev)
        assert rel_fro(got, alone) <= op_tol, f"layer {i} ({layer.name}) on its own input: {rel_fro(got, alone):.3e}"
        if layer.act == "relu6":
            assert got.min() >= 0 and got.max() <= 6
        prev = got
    check_against_oracle(host(model.layer_output(28)), probs, want[28], want[29], rel=1e-2 if math == "tf32" else 1e-4)
    model.close()


def test_config3_mobilenet_025_128(ctx, oracle):
    x, layers = si.config_mobilenet(0.25, 128, 1, seed=si.CONFIG_SEEDS["mobilenet_025_128"])
    want = oracle.run_model(layers, x, keep_all=True)
    model = ctx.model(layers, x.shape)
    model.set_keep_all(True)
    got_logits, got_probs = logits_and_probs(model, dev(x))
    ctx.check_device_status()
    check_against_oracle(got_logits, got_probs, want[-2], want[-1])
    model.close()


def test_config4_mobilenet_100_224(ctx, oracle):
    x, layers = si.config_mobilenet(1.0, 224, 1, seed=si.CONFIG_SEEDS["mobilenet_100_224"])
    want = oracle.run_model(layers, x, keep_all=True)
    model = ctx.model(layers, x.shape)
    model.set_keep_all(True)
    got_logits, got_probs = logits_and_probs(model, dev(x))
    ctx.check_device_status()
    check_against_oracle(got_logits, got_probs, want[-2], want[-1])
    # ping-pong arena and keep-all buffers give the same bits
    model.set_keep_all(False)
    assert same_bits(host(model.run(dev(x))), got_probs)
    # fp32 CUDA-core variant of the same model: tighter agreement
    ctx.set_math("fp32")
    try:
        exact = ctx.model(layers, x.shape)
    finally:
        ctx.set_math("tf32")
    exact.set_keep_all(True)
    el, ep = logits_and_probs(exact, dev(x))
    check_against_oracle(el, ep, want[-2], want[-1], rel=1e-4)
    exact.close()
    model.close()


@pytest.mark.parametrize("config", ["mobilenet_025_128", "mobilenet_100_224"])
def test_batch1_configs_under_graph_replay(ctx, oracle, config):
    """Configs 3 and 4 in the configuration whose latency the benchmark reports for batch 1: graph replay of
    the planned run (fused kernels, split-K GEMMs, programmatic dependent launch), against the oracle."""
    import torch

    alpha, hw = (0.25, 128) if config == "mobilenet_025_128" else (1.0, 224)
    x, layers = si.config_mobilenet(alpha, hw, 1, seed=si.CONFIG_SEEDS[config])
    want = oracle.run_model(layers, x, keep_all=True)
    model = ctx.model(layers, x.shape)
    xd = dev(x)
    out = torch.empty(model.output_shape, device="cuda")
    model.run(xd, out=out)  # launch by launch first (function attributes are set outside a capture)
    plain = host(out).copy()
    model.set_graph(True)
    for _ in range(3):  # the first captures, the others replay
        out.zero_()
        model.run(xd, out=out)
    got_probs = host(out)
    # the dense output is the last intermediate written: the ping-pong region still holds it
    got_logits = host(model.layer_output(model.n_layers - 2))
    ctx.check_device_status()
    assert same_bits(got_probs, plain)
    check_against_oracle(got_logits, got_probs, want[-2], want[-1])
    model.close()


def test_config5_mobilenet_100_224_batch128_all_images(ctx, oracle):
    """Full batch-128 run in the launch configuration the benchmark times, every image against the oracle."""
    import torch

    x, layers = si.config_mobilenet(1.0, 224, 128, seed=si.CONFIG_SEEDS["mobilenet_100_224_b128"])
    model = ctx.model(layers, x.shape)
    xd = dev(x)
    probs = model.run(xd)
    logits = model.layer_output(model.n_layers - 2)  # the ping-pong region still holds the dense output
    ctx.check_device_status()
    probs, logits = host(probs), host(logits)
    assert probs.shape == (128, 1000)
    assert np.all(np.abs(probs.astype(np.float64).sum(-1) - 1) <= 1e-5)
    want = oracle.run_model(layers, x, keep_all=True)
    check_against_oracle(logits, probs, want[-2], want[-1])
    # host-buffer entry point: same bits as the device-resident run
    hin = torch.from_numpy(x).pin_memory()
    hout = torch.empty(128, 1000).pin_memory()
    model.run_host(hin, hout)
    assert same_bits(hout.numpy(), probs)
    model.run_host(hin, hout.zero_())  # second call: the slices replay their captured graphs
    assert same_bits(hout.numpy(), probs)
    # asynchronous host runs: three calls in a row (the third has to wait for the first, whose staging
    # buffers it reuses), different inputs, outputs checked after one wait
    hin2 = torch.from_numpy(np.ascontiguousarray(x[::-1])).pin_memory()  # the images in reverse order
    hout2, hout3 = torch.zeros(128, 1000).pin_memory(), torch.zeros(128, 1000).pin_memory()
    hout.zero_()
    model.run_host_async(hin, hout)
    model.run_host_async(hin2, hout2)
    model.run_host_async(hin, hout3)
    model.host_wait()
    ctx.check_device_status()
    assert same_bits(hout.numpy(), probs) and same_bits(hout3.numpy(), probs)
    assert same_bits(hout2.numpy(), probs[::-1])
    # graph replay of the whole-batch run gives the same bits as launch-by-launch
    out2 = torch.empty(128, 1000, device="cuda")
    model.set_graph(True)
    model.run(xd, out=out2)
    model.run(xd, out=out2)
    assert same_bits(host(out2), probs)
    model.set_graph(False)
    # per-layer profile returns one positive time per layer
    ms = model.profile(xd, reps=2)
    assert len(ms) == 30 and all(t > 0 for t in ms)
    model.close()


def test_model_rejects_wrong_shapes(ctx, tfjsb):
    import torch

    x, layers = si.config_mobilenet(0.25, 32, 1, seed=5, classes=10)
    model = ctx.model(layers, x.shape)
    with pytest.raises(tfjsb.TfjsbError) as e:
        model.run(torch.zeros(1, 33, 32, 3, device="cuda"))
    assert e.value.status_name == "SHAPE"
    with pytest.raises(tfjsb.TfjsbError) as e:
        model.run(dev(x), out=torch.zeros(1, 11, device="cuda"))
    assert e.value.status_name == "SHAPE"
    bad = si.mobilenet_v1_layers(0.25, 10)
    si.make_model_weights(bad, 3, 5)
    bad[1].dilations = (2, 2)
    bad[1].strides = (2, 2)
    with pytest.raises(tfjsb.TfjsbError) as e:
        ctx.model(bad, x.shape)
    assert e.value.status_name == "UNSUPPORTED"
    model.close()


@pytest.mark.parametrize("batch,hw,classes", [(23, 33, 10), (25, 33, 10), (37, 32, 101), (50, 33, 7), (75, 31, 6), (97, 32, 33)])
def test_host_runs_in_uneven_slices(ctx, oracle, batch, hw, classes):
    """Batches that do not divide evenly, images and results whose size is no multiple of 16 bytes."""
    import torch

    x, layers = si.config_mobilenet(0.25, hw, batch, seed=4243, classes=classes)
    want = oracle.run_model(layers, x)
    model = ctx.model(layers, x.shape)
    hin = torch.from_numpy(x).pin_memory()
    for _ in range(3):  # launch by launch, then as graph replays, on both sets of staging buffers
        hout = torch.full(model.output_shape, -1.0).pin_memory()
        model.run_host(hin, hout)
        # probabilities in [0, 1] of a model whose logits are within 1e-2 of their range (the whole-model bar)
        assert np.max(np.abs(hout.numpy() - want)) <= 2e-2 * want.max() and np.allclose(hout.numpy().sum(-1), 1, atol=1e-5)
    ctx.check_device_status()
    model.close()


def _close_logits(got, want, rel=1e-2):
    span = want.max(-1, keepdims=True) - want.min(-1, keepdims=True)
    assert np.max(np.abs(got - want) / span) <= rel


SMALL_MODELS = [
    (1, 64, 0.25, 32), (2, 65, 0.25, 32), (3, 33, 0.5, 32), (1, 96, 0.75, 32), (5, 47, 0.25, 32), (9, 64, 0.25, 32), (17, 32, 0.25, 32), (20, 50, 0.25, 32),
    (38, 32, 0.25, 32), (60, 32, 0.25, 32), (100, 32, 0.25, 32), (2, 81, 0.25, 16), (1, 81, 0.25, 8), (40, 33, 0.25, 8)]


# (no dilation in the bfloat16 storage mode)
@pytest.mark.parametrize("batch,hw,alpha,output_stride,math",
                         [(*m, math) for math in ("tf32", "bf16") for m in SMALL_MODELS if math == "tf32" or m[3] == 32])
def test_layers_of_a_small_model_in_one_kernel(ctx, oracle, batch, hw, alpha, output_stride, math):
    """Clusters of 16 blocks down to a few, several images per cluster, odd widths, dilated layers: the layers in one
    kernel against the layers' own kernels (both at the whole-model bar from the oracle; a bfloat16 value at a rounding
    boundary may go either way, 2^-8 of it, in a layer of hundreds), and the first images against the oracle."""
    if output_stride == 32:
        x, layers = si.config_mobilenet(alpha, hw, batch, seed=4243, classes=100)
    else:
        x, layers = si.config_mobilenet_atrous(alpha, hw, batch, output_stride, seed=4243, classes=100)
    ctx.set_math(math)
    try:
        model = ctx.model(layers, x.shape)
    finally:
        ctx.set_math("tf32")
    xd, n = dev(x), len(layers)
    probs = [host(model.run(xd)) for _ in range(2)]
    one_kernel = model.layer_kernels()
    logits, pooled = host(model.layer_output(n - 2)), host(model.layer_output_f32(n - 3))
    model.set_graph(True)
    probs.append(host(model.run(xd)))
    model.set_graph(False)
    ctx.check_device_status()
    assert all(same_bits(p, probs[0]) for p in probs)
    assert np.allclose(probs[0].sum(-1), 1, atol=1e-5)
    if (alpha, hw) != (0.75, 96):
        assert one_kernel[0] == "chain_kernel", one_kernel[0]
    model.set_fusion("off")
    model.run(xd)
    assert "chain_kernel" not in model.layer_kernels()
    _close_logits(logits, host(model.layer_output(n - 2)))
    own = host(model.layer_output_f32(n - 3))
    assert rel_fro(pooled, own) <= 1e-2
    if math == "tf32":
        few = min(batch, 3)
        _close_logits(logits[:few], oracle.run_model(layers, x[:few], keep_all=True)[-2])
    model.close()


@pytest.mark.parametrize("batch", [1, 6])
def test_layers_in_one_kernel_without_bias_or_padding(ctx, oracle, batch):
    layers = si.mobilenet_v1_layers(0.25, 32)
    si.make_model_weights(layers, 3, 77)
    for i, layer in enumerate(layers):
        if i < 12 and layer.kind in ("conv2d", "depthwise_conv2d"):
            layer.pad = "valid"
        if i % 3 == 0 and layer.kind in ("conv2d", "depthwise_conv2d", "dense"):
            layer.bias = None
        if i % 5 == 1 and layer.kind in ("conv2d", "depthwise_conv2d"):
            layer.act = "none" if i % 2 else "relu"
    x = si.uniform(78, 0, (batch, 101, 79, 3), -1, 1)
    want = oracle.run_model(layers, x, keep_all=True)
    model = ctx.model(layers, x.shape)
    probs = host(model.run(dev(x)))
    assert model.layer_kernels()[0] == "chain_kernel"
    _close_logits(host(model.layer_output(len(layers) - 2)), want[-2])
    assert np.max(np.abs(probs - want[-1])) <= 2e-2 * want[-1].max()
    ctx.check_device_status()
    model.close()


def _integer_mobilenet(alpha, hw, batch, classes, tail, seed):
    """Small integers everywhere, the last layers left out: every product and sum is exact, and 2 x 2 or 4 x 4 positions
    average to quarters or sixteenths, so two orders of summation give the same bits."""
    layers = si.mobilenet_v1_layers(alpha, classes)[:tail]
    chans = si.layer_channels(layers, 3)
    for i, (layer, (cin, cout)) in enumerate(zip(layers, chans)):
        fh, fw = layer.filter_hw
        if layer.kind == "depthwise_conv2d":
            layer.filter = si.small_integers(seed, 2 * i + 1, (fh, fw, cin, 1), -1, 1)
        elif layer.kind == "conv2d":
            layer.filter = si.small_integers(seed, 2 * i + 1, (fh, fw, cin, cout), -1, 1)
        elif layer.kind == "dense":
            layer.filter = si.small_integers(seed, 2 * i + 1, (cin, cout), -2, 2)
        else:
            continue
        layer.bias = si.small_integers(seed, 2 * i + 2, (cout,), -2, 2)
    return si.small_integers(seed, 0, (batch, hw, hw, 3), -3, 3), layers


@pytest.mark.parametrize("math", ["tf32", "bf16"])
@pytest.mark.parametrize("tail", [28, 29, 30])
@pytest.mark.parametrize("batch,hw,alpha", [(1, 64, 0.25), (3, 128, 0.25), (40, 64, 0.25), (2, 64, 0.5)])
def test_outputs_that_survive_a_run_in_one_kernel(ctx, batch, hw, alpha, tail, math):
    """A model that ends in its pooled features, its logits or its probabilities: the outputs of the two layers before the
    last can be read after a run, whether the layers ran as one kernel or each as its own; both with the same bits."""
    x, layers = _integer_mobilenet(alpha, hw, batch, 12, tail, 4250)
    ctx.set_math(math)
    try:
        model = ctx.model(layers, x.shape)
    finally:
        ctx.set_math("tf32")
    xd, n = dev(x), len(layers)
    out = host(model.run(xd))
    assert model.layer_kernels()[0] == "chain_kernel"
    survivors = [host(model.layer_output_f32(i)) for i in (n - 2, n - 3)]
    ctx.check_device_status()
    model.set_fusion("off")
    want = host(model.run(xd))
    assert "chain_kernel" not in model.layer_kernels()
    for got, i in zip(survivors, (n - 2, n - 3)):
        own = host(model.layer_output_f32(i))
        assert len(np.unique(own)) > 4 and same_bits(got, own), layers[i].name
    assert np.max(np.abs(out - want)) <= 1e-6 if tail == 30 else same_bits(out, want)  # exp() is not exact
    model.close()


def test_one_kernel_models_launch_their_kernel_in_graph_mode_too(ctx):
    """A run of one kernel leaves a graph nothing to save, and costs its instantiation for every new buffer: in graph mode it
    is launched as it is.  Seen from outside: it can be recorded into a graph of the caller's, which a replay cannot."""
    import torch

    x, layers = si.config_mobilenet(0.25, 64, 2, seed=4243, classes=20)
    model = ctx.model(layers, x.shape)
    xd, out = dev(x), torch.empty(model.output_shape, device="cuda")
    model.run(xd, out=out)
    assert model.launches_per_run == 1
    plain = host(out).copy()
    model.set_graph(True)
    model.run(xd, out=out)
    assert same_bits(host(out), plain)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        model.run(xd, out=out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert same_bits(host(out), plain)
    ctx.check_device_status()
    del graph
    model.close()


@pytest.mark.parametrize("alpha,hw,batch,sliced", [(0.25, 96, 25, False), (0.25, 64, 127, False), (0.5, 64, 101, False), (0.5, 160, 127, True)])
def test_host_runs_are_sliced_only_where_copies_are_long(ctx, alpha, hw, batch, sliced):
    """Small images through small models: a slice would add its kernels' fixed times and hide next to no copying, in the
    blocking call and more so in the asynchronous one, whose copies overlap the run before.  Seen in the kernels launched."""
    import torch

    x, layers = si.config_mobilenet(alpha, hw, batch, seed=4243, classes=12)
    model = ctx.model(layers, x.shape)
    hin, hout = torch.from_numpy(x).pin_memory(), torch.zeros(model.output_shape).pin_memory()
    model.run_host(hin, hout)
    first = hout.clone()

    def launched(call):
        before = ctx.launch_count
        call(hin, hout.zero_())
        model.host_wait()
        return ctx.launch_count - before

    whole = model.launches_per_run
    blocking, asynchronous = launched(model.run_host), launched(model.run_host_async)
    assert (blocking > whole) if sliced else (blocking == asynchronous == whole)
    # the two calls may cut the batch differently: the same results up to the order of sums
    assert np.max(np.abs(hout.numpy() - first.numpy())) <= 2e-2 * float(first.max())
    ctx.check_device_status()
    model.close()


def test_a_look_at_the_layers_does_not_end_the_one_kernel_for_good(ctx):
    x, layers = si.config_mobilenet(0.25, 64, 1, seed=4243, classes=20)
    model = ctx.model(layers, x.shape)
    xd = dev(x)
    first = host(model.run(xd))
    assert model.launches_per_run == 1
    model.set_keep_all(True)
    every_layer = host(model.run(xd))
    model.set_keep_all(False)
    assert same_bits(host(model.run(xd)), every_layer) and model.launches_per_run == len(layers)
    model.set_fusion("auto")
    assert same_bits(host(model.run(xd)), first) and model.launches_per_run == 1
    model.set_keep_all(True)
    assert same_bits(host(model.run(xd)), every_layer)
    ctx.check_device_status()
    model.close()


def test_profile_of_a_model_that_runs_as_one_kernel(ctx):
    x, layers = si.config_mobilenet(0.25, 64, 1, seed=4243, classes=20)
    model = ctx.model(layers, x.shape)
    xd = dev(x)
    first = host(model.run(xd))
    ms = model.profile(xd, reps=3)
    # every layer has its time, none of them most of it
    assert len(ms) == len(layers) and min(ms) > 0 and max(ms) < 0.5 * sum(ms)
    assert same_bits(host(model.run(xd)), first) and model.layer_kernels()[0] == "chain_kernel"
    ctx.check_device_status()
    model.close()


@pytest.mark.parametrize("batch,hw,alpha", [(1, 96, 0.25), (5, 64, 0.25), (40, 64, 0.25), (2, 96, 0.5)])
def test_products_of_the_one_kernel_are_tf32_products_with_fp32_sums(ctx, oracle, batch, hw, alpha):
    """The layers that can be read after a run as one kernel, each against the oracle on the input that it had: the last
    pointwise layer at the operand-matched bar of the tensor-core kernels (operands cut to TF32, sums in another order),
    the pool and the dense layer, which are fp32 arithmetic, at the bar of the CUDA-core kernels."""
    x, layers = si.config_mobilenet(alpha, hw, batch, seed=4251, classes=52)
    features, logits = ctx.model(layers[:28], x.shape), ctx.model(layers[:29], x.shape)
    xd = dev(x)
    pooled = host(features.run(xd))
    dw, pw = (host(features.layer_output_f32(i)) for i in (25, 26))
    out = host(logits.run(xd))
    assert features.layer_kernels()[0] == logits.layer_kernels()[0] == "chain_kernel"
    seen = host(logits.layer_output_f32(27))
    ctx.check_device_status()
    own = oracle.conv2d(dw, layers[26].filter, bias=layers[26].bias, act="relu6", operand="tf32_rz")
    assert rel_fro(pw, own) <= 2e-5
    assert rel_fro(pooled, pw.astype(np.float64).mean((1, 2))) <= 1e-6
    assert rel_fro(seen, pooled) <= 1e-6  # (the two models' plans may differ)
    assert rel_fro(out, seen.astype(np.float64) @ layers[28].filter.astype(np.float64) + layers[28].bias) <= 1e-6
    features.close()
    logits.close()
