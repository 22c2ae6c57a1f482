"""The kernels for problems of few tiles (contraction split over a cluster, one-launch batch-norm, weight gradients without partial
matrices) and the ReLU masks / bias gradients that a layer's backward pass takes along for the layer below, at sizes where they can go wrong;
and the large problems' kernels at the same sizes (a context sized for one or two SMs takes those).
Tolerances are those of tests/test_gpu_bf16.py: 2e-2 (L2) and 3e-2 (element-wise) on every tensor without ReLU layers, and with
them the larger of 2e-2 and three times the oracle's own response to a one-ulp change of 0.1 % of the inputs."""
import pytest

from paper_2509_05679_b200 import synth as sy
from harness import run_parity
from test_gpu_bf16 import FAMILY_NETS, _block, _head

pytestmark = pytest.mark.gpu

LINEAR = {f"{k}-{n}": sy.mlp_layers([k, n, 64, 10]) for k, n in ((64, 64), (128, 192), (1024, 128), (704, 320))}
CONV = {
    # 3x3 on 2x2 and 4x4 images (a tile spans 32 / 8 samples), stride 2 with its four parity classes, 1x1
    "tiny-images": ((4, 4, 64), [(sy.CONV3X3, 64, 64, 1, 1), (sy.RELU, 64, 64, 1, 0), (sy.CONV3X3, 64, 128, 2, 1), (sy.RELU, 128, 128, 1, 0)] + _head(128)),
    "pointwise": ((8, 8, 64), [(sy.CONV1X1, 64, 128, 1, 1), (sy.RELU, 128, 128, 1, 0), (sy.CONV1X1, 128, 64, 1, 1), (sy.RELU, 64, 64, 1, 0)] + _head(64)),
    # conv -> ReLU -> pool, conv -> ReLU -> global average: masks and bias gradients taken along by both
    "pool-gap": ((16, 16, 64), [(sy.CONV3X3, 64, 64, 1, 1), (sy.RELU, 64, 64, 1, 0), (sy.MAXPOOL2, 64, 64, 2, 0), (sy.CONV3X3, 64, 64, 1, 1), (sy.RELU, 64, 64, 1, 0)] + _head(64)),
}


@pytest.mark.parametrize("workers,batch", [(1, 1), (1, 129), (3, 43)])
@pytest.mark.parametrize("name", sorted(LINEAR))
def test_linear_layers(orc, name, workers, batch):
    """One sample, one more than a tile, a ragged second tile; contractions of 1 to 16 steps (splits 1 to 8)."""
    layers = LINEAR[name]
    net = sy.Net(name, layers, [], 1, 1, layers[0][1], 10, workers, batch, 0.05, "bf16")
    run_parity(orc, net, 2, grad_tol=2e-2, noise_factor=3.0, loss_tol=1e-3)


@pytest.mark.parametrize("workers,batch", [(1, 2), (2, 9), (3, 16)])
@pytest.mark.parametrize("name", sorted(CONV))
def test_convolutions_with_masks_taken_along(orc, name, workers, batch):
    shape, layers = CONV[name]
    run_parity(orc, sy.Net(name, layers, [], *shape, 10, workers, batch, 0.05, "bf16"), 1, grad_tol=2e-2, noise_factor=3.0, loss_tol=1e-3)


@pytest.mark.parametrize("c", [16, 32, 48, 64, 192])
@pytest.mark.parametrize("workers,batch,size", [(1, 1, 4), (2, 9, 8), (5, 3, 16)])
def test_one_launch_batch_norm(orc, c, workers, batch, size):
    """Rows per worker from 16 (most threads idle) to 768, slices of 16, 32 and 64 channels, a residual block with its accumulations."""
    layers = [(sy.CONV3X3, 3, c, 1, 0), (sy.BATCHNORM, c, c, 1, 0)] + _block(c, c, 1) + _head(c)
    net = sy.without_relu(sy.Net("bn", layers, [], size, size, 3, 10, workers, batch, 0.05, "bf16"))
    run_parity(orc, net, 1, grad_tol=2e-2, elem_tol=3e-2, pair_bn=True, loss_tol=1e-3)


@pytest.mark.parametrize("sms", [1, 2])
@pytest.mark.parametrize("name", sorted(FAMILY_NETS))
def test_large_problem_kernels_on_small_sizes(orc, name, sms):
    shape, layers = FAMILY_NETS[name]
    net = sy.without_relu(sy.Net(name, layers, [], *shape, 10, 2, 8, 0.05, "bf16"))
    run_parity(orc, net, 1, grad_tol=2e-2, elem_tol=3e-2, pair_bn=True, loss_tol=1e-3, grid_sms=sms)


def test_masks_taken_along_by_the_large_kernels(orc):
    """3 x 43 samples on one SM's grid: the persistent kernels' epilogues mask and sum, with a ragged last tile."""
    layers = sy.mlp_layers([256, 256, 256, 10])
    net = sy.Net("mlp", layers, [], 1, 1, 256, 10, 3, 43, 0.05, "bf16")
    run_parity(orc, net, 2, grad_tol=2e-2, noise_factor=3.0, loss_tol=1e-3, grid_sms=1)
    shape, layers = CONV["pool-gap"]
    run_parity(orc, sy.Net("pool-gap", layers, [], *shape, 10, 2, 9, 0.05, "bf16"), 1, grad_tol=2e-2, noise_factor=3.0, loss_tol=1e-3, grid_sms=1)


# batch-norm as the network's first layer has no input gradient to write: general kernels (fp32; bf16 with 48 channels over 4 MB), one-launch
# kernels, streamed kernels (64 channels, 4.2 MB), with a ReLU and with a residual, whose gradients are not needed either
@pytest.mark.parametrize("dtype,c,workers,batch,size", [("fp32", 8, 2, 3, 8), ("bf16", 16, 2, 3, 8), ("bf16", 64, 2, 64, 16), ("bf16", 48, 2, 82, 16)])
@pytest.mark.parametrize("residual", [False, True])
def test_batch_norm_on_the_network_input(orc, dtype, c, workers, batch, size, residual):
    first = [(sy.BATCHNORM, c, c, 1, 0)]
    if residual:
        first = [(sy.RES_BEGIN, c, c, 1, 0)] + first + [(sy.RES_ADD, c, c, 1, 0)]
    layers = first + [(sy.CONV3X3, c, 8, 1, 1)] + _head(8)
    net = sy.Net("bn-first", layers, [], size, size, c, 10, workers, batch, 0.05, dtype)
    if dtype == "fp32":
        run_parity(orc, net, 2, param_tol=1e-5, loss_tol=1e-5)
    else:
        run_parity(orc, net, 1, grad_tol=2e-2, elem_tol=3e-2, pair_bn=True, loss_tol=1e-3)


@pytest.mark.parametrize("batch", [2048, 2049, 4737])
@pytest.mark.parametrize("hidden", [64, 320])
def test_classifier_head_of_many_samples(orc, batch, hidden):
    """64 and 65 blocks of 32 samples (the line between the two ways of adding their partial gradients), and 149 (all columns in one block), with 8 and 40
    vectors of columns; the masked error and the bias gradient that the head takes along for the layer below."""
    net = sy.Net("mlp", sy.mlp_layers([64, hidden, 10]), [], 1, 1, 64, 10, 1, batch, 0.05, "bf16")
    run_parity(orc, net, 1, grad_tol=2e-2, noise_factor=3.0, loss_tol=1e-3)
