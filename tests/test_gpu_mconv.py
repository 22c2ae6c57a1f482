"""The convolutions of 16-multiple channel counts off the TMA path, on both sides of the line between the tensor-core kernels (mconv.cu) and the packed-FMA kernels,
at the edges of their tiles: images of odd sides, of one row or column, smaller than a tile; strides 1 and 2, 3x3 and 1x1; one, two and three blocks of 16
channels; batches that leave a tile ragged; magnitudes far from 1, where the parts of a split value get small.  One step of ReLU-free networks against the
oracle, with the tolerances of tests/test_gpu_fconv.py.  TAKEN: shapes whose three passes all run on mconv.cu, which the profiler has to say."""
import time

import numpy as np
import pytest

from paper_2509_05679_b200 import synth as sy
from harness import make_ctx, make_oracle, max_rel_err, run_parity

pytestmark = pytest.mark.gpu

# (H, W), first layer's width, kind, second layer's width, stride
SHAPES = [((5, 7), 16, sy.CONV3X3, 48, 1), ((33, 9), 16, sy.CONV3X3, 16, 1), ((16, 1), 16, sy.CONV3X3, 32, 1), ((2, 2), 32, sy.CONV3X3, 16, 1), ((6, 10), 32, sy.CONV3X3, 64, 2),
          ((14, 14), 16, sy.CONV3X3, 32, 2), ((7, 11), 16, sy.CONV1X1, 32, 1), ((6, 10), 48, sy.CONV1X1, 16, 2), ((4, 4), 80, sy.CONV3X3, 96, 1)]

ALL, EVEN, ONE = [(1, 1), (3, 9), (2, 70)], [(1, 1), (2, 70)], [(1, 1)]
# and the workers x batches that are taken with fp32 storage (bf16: all three); 16x16, 15x13 and 4x64: 2 x 70 with 32 output channels a CTA
TAKEN = [(((12, 20), 16, sy.CONV3X3, 16, 1), ALL), (((33, 9), 16, sy.CONV3X3, 16, 1), EVEN), (((1, 40), 48, sy.CONV3X3, 16, 1), ONE), (((7, 7), 48, sy.CONV3X3, 32, 1), ALL),
         (((15, 13), 32, sy.CONV3X3, 32, 1), ALL), (((16, 16), 32, sy.CONV3X3, 32, 1), ALL), (((4, 4), 80, sy.CONV3X3, 96, 1), ALL), (((14, 14), 16, sy.CONV3X3, 32, 2), ALL),
         (((16, 30), 32, sy.CONV3X3, 48, 2), ALL), (((6, 10), 32, sy.CONV3X3, 64, 2), ONE), (((4, 64), 32, sy.CONV1X1, 32, 1), ALL), (((2, 64), 16, sy.CONV1X1, 32, 2), ALL)]


def _net(shape, dtype, workers, batch, bn):
    (h, w), c, kind, co, stride = shape
    norm = lambda n: [(sy.BATCHNORM, n, n, 1, 0)] if bn else []
    bias = 0 if bn else sy.FLAG_BIAS
    layers = [(sy.CONV3X3, 3, c, 1, bias)] + norm(c) + [(kind, c, co, stride, bias)] + norm(co) + [(sy.GLOBAL_AVGPOOL, co, co, 1, 0), (sy.LINEAR, co, 10, 1, 1)]
    return sy.Net("mconv", layers, [], h, w, 3, 10, workers, batch, 0.05, dtype)


def _id(s):
    return f"{s[0][0]}x{s[0][1]}-{s[1]}-{s[3]}-k{3 if s[2] == sy.CONV3X3 else 1}-s{s[4]}"


def _assert_taken(net, shape):
    """Forward, input gradient and weight gradient of the second layer ran on mconv.cu."""
    import torch
    from paper_2509_05679_b200 import binding
    ctx = make_ctx(net, sy.init_params(net.layers, 0))
    try:
        ctx.profile(True)
        ctx.step(binding.to_device(net.dtype, sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda())
        ran = {k for k in ctx.profile_read() if k.startswith(("mma_", "fma_"))}
    finally:
        ctx.close()
    (h, w), c, kind, co, stride = shape
    tag = f"[{h}x{w} {c}->{co} k{3 if kind == sy.CONV3X3 else 1} s{stride}]"
    assert {k for k in ran if k.endswith(tag)} == {f"mma_{p}{tag}" for p in ("fwd", "dgrad", "wgrad")}, ran


@pytest.mark.parametrize("shape,workers,batch", [(s, w, b) for s, sizes in TAKEN for w, b in sizes], ids=lambda v: _id(v) if isinstance(v, tuple) else str(v))
def test_fp32_on_tensor_cores(orc, shape, workers, batch):
    net = _net(shape, "fp32", workers, batch, False)
    _assert_taken(net, shape)
    run_parity(orc, net, 1, param_tol=1e-5, loss_tol=1e-5, grad_tol=1e-5)
    run_parity(orc, _net(shape, "fp32", workers, batch, True), 1, param_tol=1e-5, loss_tol=1e-5)


@pytest.mark.parametrize("workers,batch", EVEN)
@pytest.mark.parametrize("shape", [s for s, _ in TAKEN if s[0] != (6, 10)], ids=_id)
def test_bf16_on_tensor_cores(orc, shape, workers, batch):
    terms = shape[1] * (9 if shape[2] == sy.CONV3X3 else 1)
    net = _net(shape, "bf16", workers, batch, False)
    _assert_taken(net, shape)
    run_parity(orc, net, 1, grad_tol=2e-3 if terms <= 144 and workers * batch in (1, 2, 4, 8) else 2e-2, loss_tol=1e-4)


@pytest.mark.parametrize("workers,batch", [(1, 1), (3, 9), (2, 70)])
@pytest.mark.parametrize("shape", SHAPES, ids=_id)
def test_fp32(orc, shape, workers, batch):
    run_parity(orc, _net(shape, "fp32", workers, batch, False), 1, param_tol=1e-5, loss_tol=1e-5, grad_tol=1e-5)
    run_parity(orc, _net(shape, "fp32", workers, batch + 1, True), 1, param_tol=1e-5, loss_tol=1e-5)


@pytest.mark.parametrize("workers,batch", [(1, 1), (2, 9)])
@pytest.mark.parametrize("shape", SHAPES, ids=_id)
def test_bf16_storage(orc, shape, workers, batch):
    terms = shape[1] * (9 if shape[2] == sy.CONV3X3 else 1)
    run_parity(orc, _net(shape, "bf16", workers, batch, False), 1, grad_tol=2e-3 if terms <= 144 and workers * batch in (1, 2, 4, 8) else 2e-2, loss_tol=1e-4)


@pytest.mark.parametrize("exponent", [-124, -110, -60, 40, 100, 122])
def test_values_far_from_one(orc, exponent):
    """First layer's weights times 2^exponent, second layer's divided by it: the second layer's inputs are that far from 1, its outputs as before; the
    scalings are exact (2^-122: to 2^-23), so gradients are compared as scaled.  From 2^111 on a split value has infinite parts and its products are computed one by one; down
    to the smallest normal number nothing is lost.  Gradients that fp32 itself cannot hold (of the second layer at 2^-124, of the first at 2^122) are left out."""
    import torch
    from paper_2509_05679_b200 import binding
    net = _net(((9, 8), 16, sy.CONV3X3, 32, 1), "fp32", 2, 5, False)
    p0 = sy.init_params(net.layers, 0)
    n1 = 16 * 27
    p0[n1:n1 + 16] = 0.0
    scaled = p0.copy()
    scaled[:n1] = np.ldexp(p0[:n1], exponent)
    n2 = n1 + 16 + 32 * 9 * 16
    scaled[n1 + 16:n2] = np.ldexp(p0[n1 + 16:n2], -exponent)
    x, y = sy.batch_inputs(net, 0), sy.batch_labels(net, 0)
    o = make_oracle(orc, net, p0)
    o.step(x, y, 0.0)
    g = np.mean([o.grads(s) for s in range(net.n_workers)], axis=0)
    ctx = make_ctx(net, scaled)
    try:
        ctx.set_lr(0.0)
        ctx.step(binding.to_device("fp32", x), torch.from_numpy(y).cuda())
        got = np.asarray(ctx.grads(), np.float64)
    finally:
        ctx.close()
    got[:n1 + 16] = np.ldexp(got[:n1 + 16], exponent)          # d/d(w 2^e) = 2^-e d/dw
    got[n1 + 16:n2] = np.ldexp(got[n1 + 16:n2], -exponent)
    if exponent < -120:
        got[n1 + 16:n2] = g[n1 + 16:n2]
    if exponent > 120:
        got[:n1 + 16] = g[:n1 + 16]
    err, where = max_rel_err(got, g, net.layers)
    assert err <= 1e-5, (err, where)


@pytest.mark.parametrize("stride", [1, 2])
@pytest.mark.parametrize("at", ["weight looked at", "weight", "pixel", "infinite weight"])
def test_nan_where_packed_fma_has_it(at, stride):
    """One NaN (or infinity) among the second layer's weights or in the input: the gradients that are NaN, and the values of the others, are those of kernel_path 1.
    ReLU turns NaN to 0, so that the loss is finite.  1e-5 of a tensor's largest: the tolerance of test_fp32."""
    import torch
    from paper_2509_05679_b200 import binding
    layers = [(sy.CONV3X3, 16, 16, 1, 0), (sy.RELU, 16, 16, 1, 0), (sy.CONV3X3, 16, 32, stride, 0), (sy.RELU, 32, 32, 1, 0), (sy.GLOBAL_AVGPOOL, 32, 32, 1, 0), (sy.LINEAR, 32, 10, 1, 1)]
    net = sy.Net("mconv", layers, [], 16, 16, 16, 10, 2, 9, 0.0, "fp32")
    p0, x = sy.init_params(layers, 0), sy.batch_inputs(net, 0)
    w2 = p0[2304:2304 + 4608].reshape(32, 9, 16)
    if at == "weight looked at":
        w2[3, 4, 0] = np.nan
    elif at == "weight":
        w2[30, 8, 13] = np.nan
    elif at == "infinite weight":
        w2[17, 2, 5] = np.inf
    else:
        x.reshape(18, 16, 16, 16)[7, 5, 9, 11] = np.nan
    g = []
    for path in (0, 1):
        ctx = make_ctx(net, p0, kernel_path=path)
        try:
            ctx.step(binding.to_device("fp32", x), torch.from_numpy(sy.batch_labels(net, 0)).cuda())
            g.append(np.asarray(ctx.grads(), np.float64))
        finally:
            ctx.close()
    assert np.array_equal(np.isnan(g[0]), np.isnan(g[1])) and not np.isnan(g[0]).all()
    for a, b in zip(*(np.split(v, [2304, 2304 + 4608, 2304 + 4608 + 320]) for v in g)):
        ok = np.isfinite(b)
        assert np.abs(a - b)[ok].max(initial=0) <= 1e-5 * np.abs(b)[ok].max(initial=0)


def test_nan_everywhere_costs_little():
    """A diverged run goes on at its pace: less than three times as long with NaN for all parameters (12 times without the look at an output's operands, 1.4 with it)."""
    import torch
    from paper_2509_05679_b200 import binding
    layers = [(sy.CONV3X3, 3, 16, 1, 0)] + [(sy.CONV3X3, 16, 16, 1, 0)] * 8 + [(sy.CONV3X3, 16, 32, 2, 0), (sy.CONV3X3, 32, 32, 1, 0), (sy.GLOBAL_AVGPOOL, 32, 32, 1, 0), (sy.LINEAR, 32, 10, 1, 1)]
    net = sy.Net("mconv", layers, [], 32, 32, 3, 10, 4, 48, 0.0, "fp32")
    x, y = binding.to_device("fp32", sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda()
    p0, ms = sy.init_params(layers, 0), []
    for p in (p0, np.full_like(p0, np.nan)):
        ctx = make_ctx(net, p)
        try:
            for _ in range(5):
                ctx.step(x, y)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(20):
                ctx.step(x, y)
            torch.cuda.synchronize()
            ms.append((time.perf_counter() - t0) * 50)
        finally:
            ctx.close()
    assert ms[1] < 3 * ms[0], ms


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_nothing_is_laid_out_for_other_kernels(dtype):
    """Images of one pixel are left to the packed-FMA kernels: as much device memory and as many launches as with kernel_path 1.  Of images of 16x16 in the first layer only the
    forward pass reads laid-out weights (nobody wants the network's input gradient): one launch more per iteration than there."""
    import torch
    from paper_2509_05679_b200 import binding
    used = {}
    for side in (1, 16):
        layers = [(sy.CONV3X3, 16, 32, 1, 0), (sy.GLOBAL_AVGPOOL, 32, 32, 1, 0), (sy.LINEAR, 32, 10, 1, 1)]
        net = sy.Net("mconv", layers, [], side, side, 16, 10, 2, 24, 0.05, dtype)
        x, y = binding.to_device(dtype, sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda()
        for path in (0, 1):
            ctx = make_ctx(net, sy.init_params(layers, 0), kernel_path=path)
            try:
                ctx.step(x, y)
                before = ctx.stats()[1]
                for _ in range(3):
                    ctx.step(x, y)
                used[side, path] = (ctx.stats()[0], ctx.stats()[1] - before)
            finally:
                ctx.close()
    assert used[1, 0] == used[1, 1], used
    assert used[16, 0][1] == used[16, 1][1] + 3, used


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("path", [0, 1])
def test_kernel_classes(dtype, path):
    """A layer of 16-multiple channels is counted under the tensor-core classes, one of 24 channels, and everything with kernel_path 1, under those of packed FMA."""
    import torch
    from paper_2509_05679_b200 import binding
    layers = [(sy.CONV3X3, 32, 32, 1, 0), (sy.CONV3X3, 32, 32, 1, 0), (sy.CONV3X3, 32, 24, 1, 0), (sy.GLOBAL_AVGPOOL, 24, 24, 1, 0), (sy.LINEAR, 24, 10, 1, 1)]
    net = sy.Net("mconv", layers, [], 16, 16, 32, 10, 2, 24, 0.05, dtype)
    ctx = make_ctx(net, sy.init_params(layers, 0), kernel_path=path)
    try:
        ctx.profile(True)
        ctx.step(binding.to_device(dtype, sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda())
        n = {k: v["launches"] for k, v in ctx.profile_read().items() if "[" not in k}
    finally:
        ctx.close()
    tensor, fma = ({"mma_fwd": 2, "mma_dgrad": 1, "mma_wgrad": 2}, {"fma_fwd": 1, "fma_dgrad": 1, "fma_wgrad": 1}) if path == 0 else ({}, {"fma_fwd": 3, "fma_dgrad": 2, "fma_wgrad": 3})
    fma["fma_wgrad"] += 1                        # the classifier's backward pass
    assert {k: v for k, v in n.items() if k.startswith(("mma_", "fma_"))} == {**tensor, **fma}, n


def test_more_layers_than_one_launch_lays_out():
    """50 layers: the weights of 48 in one launch, of the others in a second.  Gradients beside those of the packed-FMA kernels (1e-4 in the 2-norm: roundings of
    1e-7 through 50 layers, times 20 for the last ones' cancellations)."""
    import torch
    from paper_2509_05679_b200 import binding
    layers = [(sy.CONV3X3, 16, 16, 1, 0)] * 50 + [(sy.GLOBAL_AVGPOOL, 16, 16, 1, 0), (sy.LINEAR, 16, 10, 1, 1)]
    net = sy.Net("mconv", layers, [], 8, 8, 16, 10, 2, 3, 0.0, "fp32")
    p0 = sy.init_params(layers, 0) * np.float32(0.7)           # gain of about 1 a layer
    x, y = binding.to_device("fp32", sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda()
    g = []
    for path in (0, 1):
        ctx = make_ctx(net, p0, kernel_path=path)
        try:
            if path == 0:
                ctx.profile(True)
            ctx.step(x, y)
            if path == 0:
                assert ctx.profile_read()["mma_fwd"]["launches"] == 50
            g.append(np.asarray(ctx.grads(), np.float64))
        finally:
            ctx.close()
    for a, b in zip(np.split(g[0][:50 * 2304], 50), np.split(g[1][:50 * 2304], 50)):
        assert 0 < np.linalg.norm(b) < np.inf and np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)
