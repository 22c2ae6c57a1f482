"""The packed-FMA convolutions (fconv.cu) and the fp32 batch-norm (bnorm.cu) at sizes where their tilings can go wrong: images that
are no power of two, smaller than a tile or one pixel wider, channel counts that are no multiple of 16 or of 4, strides 1 and 2, 3x3 and
1x1, batches that leave a pixel tile ragged.  ReLU-free networks (no kinks), one step against the oracle: loss, every gradient and
the updated parameters; with kernel_path 1, which keeps channels that are multiples of 16 on these kernels, and as they run without.  Tolerances: the fp32 path's 1e-5 (tests/harness.py: max_rel_err) on parameters and, in the 2-norm, on
gradients; the bf16 storage model's 2e-3 of tests/test_gpu_bf16.py for contractions of at most 144 terms and its 2e-2 beyond."""
import pytest

from paper_2509_05679_b200 import synth as sy
from harness import run_parity

pytestmark = pytest.mark.gpu

# (H, W), first layer's width, kind, second layer's width, stride
SHAPES = [((5, 7), 3, sy.CONV3X3, 5, 1), ((12, 20), 20, sy.CONV3X3, 24, 1), ((33, 9), 16, sy.CONV3X3, 8, 1), ((4, 4), 24, sy.CONV3X3, 40, 1),
          ((2, 2), 8, sy.CONV3X3, 16, 1), ((6, 10), 18, sy.CONV3X3, 16, 2), ((32, 32), 16, sy.CONV3X3, 32, 2), ((16, 16), 32, sy.CONV1X1, 64, 2),
          ((7, 11), 6, sy.CONV1X1, 12, 1), ((8, 8), 64, sy.CONV3X3, 64, 1), ((16, 1), 4, sy.CONV3X3, 16, 1)]


def _net(shape, dtype, workers, batch, bn):
    (h, w), c, kind, co, stride = shape
    norm = lambda n: [(sy.BATCHNORM, n, n, 1, 0)] if bn else []
    bias = 0 if bn else sy.FLAG_BIAS
    layers = [(sy.CONV3X3, 3, c, 1, bias)] + norm(c) + [(kind, c, co, stride, bias)] + norm(co) + [(sy.GLOBAL_AVGPOOL, co, co, 1, 0), (sy.LINEAR, co, 10, 1, 1)]
    return sy.Net("fconv", layers, [], h, w, 3, 10, workers, batch, 0.05, dtype)


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("bn", [False, True])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0][0]}x{s[0][1]}-{s[1]}-{s[3]}-k{3 if s[2] == sy.CONV3X3 else 1}-s{s[4]}")
def test_fp32(orc, shape, bn, path):
    # per-channel sums of normalised values cancel: with batch-norm in front of the average pool only the parameters have a scale of their own
    run_parity(orc, _net(shape, "fp32", 3, 5, bn), 2, param_tol=1e-5, loss_tol=1e-5, grad_tol=None if bn else 1e-5, kernel_path=path)


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: f"{s[0][0]}x{s[0][1]}-{s[1]}-{s[3]}-k{3 if s[2] == sy.CONV3X3 else 1}-s{s[4]}")
def test_bf16_storage(orc, shape, path):
    terms = shape[1] * (9 if shape[2] == sy.CONV3X3 else 1)
    run_parity(orc, _net(shape, "bf16", 2, 4, False), 1, grad_tol=2e-3 if terms <= 144 else 2e-2, loss_tol=1e-4, kernel_path=path)


@pytest.mark.parametrize("workers,batch,groups", [(4, 3, 0), (4, 20, 2), (2, 70, 0)])
@pytest.mark.parametrize("size,stride", [((7, 7), 1), ((14, 14), 2), ((9, 9), 1), ((3, 3), 1), ((6, 10), 2), ((33, 9), 1)], ids=str)
def test_images_that_no_power_of_two_covers(orc, size, stride, workers, batch, groups):
    """Tiles that reach over the image's edge, for few and for many images of one worker; windows of the batch are cut into other tiles than the whole."""
    run_parity(orc, _net((size, 16, sy.CONV3X3, 24, stride), "fp32", workers, batch, True), 1, param_tol=1e-5, loss_tol=1e-5, worker_groups=groups)


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("workers,batch", [(1, 1), (2, 130), (5, 3)])
def test_batch_sizes(orc, workers, batch, path):
    run_parity(orc, _net(((8, 8), 16, sy.CONV3X3, 32, 2), "fp32", workers, batch, True), 2, param_tol=1e-5, loss_tol=1e-5, kernel_path=path)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("batch", [74, 75])
def test_pixels_per_thread(orc, dtype, batch):
    """2 x 74 and 2 x 75 images of 8x8, 16 -> 64 channels: 296 CTAs of two pixels a thread, 300 of four (kernel_path 1: without, mconv.cu takes them)."""
    net = _net(((8, 8), 16, sy.CONV3X3, 64, 1), dtype, 2, batch, dtype == "fp32")
    if dtype == "fp32":
        run_parity(orc, net, 1, param_tol=1e-5, loss_tol=1e-5, kernel_path=1)
    else:
        run_parity(orc, net, 1, grad_tol=2e-2, loss_tol=1e-4, kernel_path=1)


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
def test_replicas_in_one_launch_equal_the_single_copy_path(dtype):
    """With P = (1/N) 1 1^T given explicitly every worker has its own weights and gradients; convolutions, batch-norm and linear layers run
    once for all of them.  Same weights as the single-copy path up to the rounding of another summation order, relative to what the
    steps changed (fp32: 1e-4, ten steps' roundings of 1e-6 with a margin; bf16 storage: the 2e-2 of the bf16 gradients)."""
    import numpy as np
    import torch
    from paper_2509_05679_b200 import binding
    layers, bs = sy.resnet_layers(widths=(8, 16), blocks=1)
    net = sy.without_relu(sy.Net("replicas", layers, [bs[0], bs[1]], 8, 8, 3, 10, 3, 5, 0.05, dtype))
    p0 = sy.perturb_params(sy.init_params(net.layers, 0, bf16=dtype == "bf16"), net.layers, 7, 0.1)
    kw = dict(dtype=dtype, in_shape=(8, 8, 3), num_classes=10)
    a = binding.Context(net.layers, net.splits, 3, 5, net.lr, mixing=np.full((3, 3), 1.0 / 3), **kw)
    b = binding.Context(net.layers, net.splits, 3, 5, net.lr, kernel_path=1, **kw)
    for c in (a, b):
        c.set_params(p0)
    for t in range(2 * net.K + 3):
        x, y = binding.to_device(dtype, sy.batch_inputs(net, t)), torch.from_numpy(sy.batch_labels(net, t)).cuda()
        for c in (a, b):
            c.step(x, y)
            c.wait_ingest()
    pb = b.params()
    for s in range(3):
        err = np.linalg.norm(a.params_worker(s) - pb) / np.linalg.norm(pb - p0)          # of what the steps changed
        assert err <= (1e-4 if dtype == "fp32" else 2e-2), (s, err)
    a.close(); b.close()
