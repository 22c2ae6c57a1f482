"""Workloads that stand for what this library is used for: training a network, split into K modules and fed by N
data-parallel workers, with fdg_step / fdg_step_host, and reading the weights.

A case is one network, one split, one batch shape and one precision; a pass is an interval of a training run between two
reads of the weights (an evaluation, a checkpoint): `steps` iterations on batches that rotate over a pool, then fdg_params.
The pipeline is full when the first pass starts (2K - 2 iterations are part of the preparation, as they are of any run),
and every pass goes on from the weights the one before it left.

Step sizes are those of the late phases of the paper's Strategy II (0.001 and the like): every case keeps a finite loss for
as long as it is run, and rounding differences stay small enough to compare two runs.
The networks and batch shapes are those of `synth.config` and of the tests; `draw` takes others of the same families.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2509_05679_b200 import binding, synth as sy

POOL = 4                # distinct batches a pass rotates over


def _case(name, family, **kw):
    c = dict(name=name, family=family, dtype="bf16", K=4, workers=4, batch=128, image=32, mixing=False, host=False, steps=20, lr=0.002)
    c.update(kw)
    return c


def listed():
    return [
        # A toy-sized network on 21 samples: the smallest call.  Nothing but launches and their latency.
        _case("mlp-ragged-fp32", "mlp", dtype="fp32", K=4, workers=3, batch=7, sizes="70-33-65-17-5", steps=100),
        # synth.config(0): the small fp32 MLP on flattened 32x32x3 images, two modules, 2 workers x 32.
        _case("mlp-fp32-K2", "mlp", dtype="fp32", K=2, workers=2, batch=32, sizes="3072-512-256-10", steps=100),
        # synth.config(1): nine linear layers of width 1024, four modules, 4 workers x 128.
        _case("mlp-bf16-K4", "mlp", K=4, workers=4, batch=128, sizes="3072" + "-1024" * 8 + "-10", steps=100),
        # synth.config(2): VGG-shaped, convolutions with bias and ReLU, max-pools, no normalisation.
        _case("vgg-bf16-K4", "vgg", K=4, workers=4, batch=128, lr=0.005),
        # synth.config(3): the headline workload, ResNet-18-shaped, four modules, 8 workers x 128, inputs in device memory.
        _case("resnet18-bf16-K4", "resnet18", K=4, workers=8, batch=128),
        # The same fed from pinned host memory with the loss read every iteration: a training loop that logs.
        _case("resnet18-bf16-K4-host", "resnet18", K=4, workers=8, batch=128, host=True),
        # The network of synth.config(4), eight modules (the longest delays), at a per-worker batch that is no power of two.
        _case("resnet18-bf16-K8", "resnet18", K=8, workers=16, batch=50),
        # The same network on a small batch: fine-tuning, or many small workers; launches and latency count.
        _case("resnet18-bf16-K4-small", "resnet18", K=4, workers=2, batch=9, steps=50, lr=0.001),
        # The paper's experiment (Sec. 5): ResNet-20, 4 workers x 48, fp32; without and with decoupling.
        _case("resnet20-fp32-K1", "resnet20", dtype="fp32", K=1, workers=4, batch=48),
        _case("resnet20-fp32-K2", "resnet20", dtype="fp32", K=2, workers=4, batch=48),
        # The same in bf16 storage.
        _case("resnet20-bf16-K2", "resnet20", dtype="bf16", K=2, workers=4, batch=48),
        # The paper's general method: one replica per worker, mixed over a ring (Eq. weight_matrix, alpha = 0.3).
        _case("resnet20-fp32-K2-ring", "resnet20", dtype="fp32", K=2, workers=4, batch=48, mixing=True),
    ]


def _log_int(rng, lo, hi):
    """An integer in lo..hi, uniform over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random):
    family = rng.choice(["mlp", "mlp", "vgg", "resnet18", "resnet18", "resnet20", "resnet20"])
    if family == "mlp":
        dtype = rng.choice(["fp32", "bf16"])
        depth = rng.randint(3, 9)
        # bf16 networks are built in widths that suit tensor cores; fp32 ones come in any
        hidden = [64 * _log_int(rng, 2, 16) if dtype == "bf16" else _log_int(rng, 17, 512) for _ in range(depth - 1)]
        sizes = [rng.choice([784, 3072]) if dtype == "bf16" else _log_int(rng, 70, 3072)] + hidden + [rng.choice([5, 10])]
        return dict(family=family, dtype=dtype, K=rng.randint(1, min(4, depth)), workers=rng.randint(1, 4), batch=_log_int(rng, 7, 128), image=32,
                    mixing=False, host=rng.random() < 0.3, sizes="-".join(map(str, sizes)), steps=100, lr=0.002)
    c = dict(family=family, dtype="bf16", image=32, mixing=False, host=rng.random() < 0.3, steps=20, lr=0.001)
    if family == "vgg":
        c.update(K=rng.randint(1, 4), workers=rng.randint(1, 4), batch=_log_int(rng, 4, 128), image=rng.choice([16, 32]))
    elif family == "resnet18":
        c.update(K=rng.choice([1, 2, 4, 8]), workers=rng.randint(1, 8), batch=_log_int(rng, 4, 100), image=rng.choice([16, 32]))
    else:
        c.update(K=rng.randint(1, 3), workers=rng.randint(2, 4), batch=_log_int(rng, 6, 48), dtype=rng.choice(["fp32", "bf16"]))
        c["mixing"] = c["dtype"] == "fp32" and rng.random() < 0.4
    return c


def _net(case) -> sy.Net:
    """Layer list and split points: modules of nearly equal numbers of weighted layers (MLP) or blocks."""
    K, s = case["K"], case["image"]
    if case["family"] == "mlp":
        sizes = [int(v) for v in case["sizes"].split("-")]
        layers = sy.mlp_layers(sizes)
        starts, shape = [2 * j for j in range(len(sizes) - 1)], (1, 1, sizes[0])
    elif case["family"] == "vgg":
        layers, starts = sy.vgg_layers()
        shape = (s, s, 3)
    else:
        layers, starts = sy.resnet_layers() if case["family"] == "resnet18" else sy.resnet_layers(widths=(16, 32, 64), blocks=3)
        starts[0], shape = 0, (s, s, 3)                    # the first layer belongs to the first block's module
    classes = layers[-1][2]
    splits = [starts[k * len(starts) // K] for k in range(1, K)]
    return sy.Net(case["family"], layers, splits, *shape, classes, case["workers"], case["batch"], case["lr"], case["dtype"])


def _ring(n):
    """Weight matrix of a ring of n workers (Sec. 2.3, Eq. weight_matrix)."""
    P = np.zeros((n, n))
    for i in range(n):
        P[i, (i + 1) % n] = P[(i + 1) % n, i] = 0.3
    return P + np.diag(1.0 - P.sum(1))


def prepare(case, seed):
    net = _net(case)
    dtype = torch.bfloat16 if net.dtype == "bf16" else torch.float32
    g = torch.Generator(device="cuda").manual_seed(seed)
    xs = [torch.randn((net.M, net.in_h, net.in_w, net.in_c), generator=g, device="cuda").to(dtype) for _ in range(POOL)]
    ys = [torch.randint(0, net.classes, (net.M,), generator=g, device="cuda", dtype=torch.int32) for _ in range(POOL)]
    if case["host"]:
        xs, ys = [x.cpu().pin_memory() for x in xs], [y.cpu().pin_memory() for y in ys]
    torch.cuda.synchronize()
    ctx = binding.Context(net.layers, net.splits, net.n_workers, net.batch, net.lr, dtype=net.dtype, in_shape=(net.in_h, net.in_w, net.in_c),
                          num_classes=net.classes, mixing=_ring(net.n_workers) if case["mixing"] else None)
    ctx.set_params(sy.init_params(net.layers, seed, bf16=net.dtype == "bf16"))
    state = dict(ctx=ctx, xs=xs, ys=ys, t=0, case=case)
    _steps(state, 2 * net.K - 2)
    torch.cuda.synchronize()
    return state


def _steps(state, n):
    """n iterations; the losses: of every iteration from host memory, of the last one otherwise."""
    ctx, xs, ys, t = state["ctx"], state["xs"], state["ys"], state["t"]
    losses = []
    if state["case"]["host"]:
        for i in range(t, t + n):
            losses.append(ctx.step_host(xs[i % POOL], ys[i % POOL], want_loss=True))
    else:
        for i in range(t, t + n):
            loss = ctx.step(xs[i % POOL], ys[i % POOL], want_loss=i == t + n - 1)
        if n:
            losses.append(loss)
    state["t"] = t + n
    return losses


def run(state):
    ctx, case = state["ctx"], state["case"]
    losses = np.array(_steps(state, case["steps"]))
    if case["mixing"]:
        return {"loss": losses, "params": [ctx.params_worker(s) for s in range(case["workers"])]}
    return {"loss": losses, "params": ctx.params()}


def work(case):
    """Per iteration: the batch and the labels read once, the fp32 weights read and written once, the layers' multiply-adds
    forward and backward (no input gradient for the first layer)."""
    net = _net(case)
    P = sy.param_count(net.layers) * (net.n_workers if case["mixing"] else 1)
    step_bytes = net.M * (net.in_elems * (2 if net.dtype == "bf16" else 4) + 4) + 8.0 * P
    return {"bytes": case["steps"] * step_bytes, "flops": case["steps"] * net.M * sy.flops_per_sample(net)}


def tolerance(case):
    """Of the weights and losses after up to three passes (60 to 300 iterations).  A correct implementation that only adds in
    another order is this far off at the most, because a ReLU input within rounding of zero switches a gradient term
    on or off and later iterations carry that on: measured by moving every initial weight by one part in 2^24, up to
    2e-4 of the weights' norm in fp32 (a flipped unit of a small MLP; 2e-5 for the convolutional networks) and, with bf16
    storage, 2e-3 of the weights' norm and 6e-3 of a small loss.  A single weight can be off by more than the
    norm: an update that is missing terms is larger than it is in the mean."""
    return {"rel": 1e-2, "max": 0.1} if case["dtype"] == "bf16" else {"rel": 1e-3, "max": 2e-2}
