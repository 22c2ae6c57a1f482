"""Steady-state iterations run as CUDA graphs whose kernels' parameters are refreshed (one graph per module, or two for
networks with more work per step).  They must do what the kernel-by-kernel enqueuing does: bit-identical weights whatever
the source of the inputs, whenever that source changes, and with profiling (which switches graphs off) in between; an input buffer
may be overwritten as soon as fdg_wait_ingest returns; a new fdg_set_params starts over."""
import numpy as np
import pytest

from paper_2509_05679_b200 import synth as sy
from harness import make_ctx

pytestmark = pytest.mark.gpu


def nets():
    small = sy.Net("mlp", sy.mlp_layers([70, 33, 65, 17, 5]), [2, 4, 6], 1, 1, 70, 5, 3, 7, 0.05, "fp32")      # one graph per module
    one = sy.Net("mlp-k1", sy.mlp_layers([40, 32, 10]), [], 1, 1, 40, 10, 2, 9, 0.05, "fp32")                  # a single module
    layers, bs = sy.resnet_layers(widths=(16, 32, 64), blocks=1)
    large = sy.Net("resnet", layers, [bs[1], bs[2]], 32, 32, 3, 10, 4, 48, 0.05, "bf16")                       # two graphs per module
    return {"small": small, "one": one, "large": large}


def _run(net, p0, steps, how, reset_at=None, **kw):
    """how(t) -> 'device', 'host' or 'profile' (device inputs, kernel by kernel)."""
    import torch
    ctx = make_ctx(net, p0, **kw)
    dt = torch.bfloat16 if net.dtype == "bf16" else torch.float32
    xb = torch.empty((net.M, net.in_h, net.in_w, net.in_c), dtype=dt, device="cuda")        # ONE buffer, overwritten before every step
    yb = torch.empty(net.M, dtype=torch.int32, device="cuda")
    losses = []
    for t in range(steps):
        if t == reset_at:
            ctx.set_params(p0)
        x, y = torch.from_numpy(sy.batch_inputs(net, t)).to(dt), torch.from_numpy(sy.batch_labels(net, t))
        if how(t) == "host":
            losses.append(ctx.step_host(x.pin_memory(), y.pin_memory(), want_loss=True))
            ctx.wait_ingest()
            continue
        xb.copy_(x); yb.copy_(y)
        torch.cuda.current_stream().synchronize()
        if how(t) == "profile":
            ctx.profile(True)
        losses.append(ctx.step(xb, yb, want_loss=t % 3 == 0))
        ctx.wait_ingest()
        if how(t) == "profile":
            ctx.profile(False)
    out = ctx.params(), ctx.grads(), [np.nan if l is None else l for l in losses]
    ms = ctx.module_times()
    ctx.close()
    assert np.all(ms > 0)
    return out


@pytest.mark.parametrize("name", ["small", "one", "large"])
def test_sources_and_interruptions_do_not_change_the_weights(name):
    net = nets()[name]
    p0 = sy.perturb_params(sy.init_params(net.layers, 0, bf16=net.dtype == "bf16"), net.layers, 7, 0.1)
    steps = 4 * net.K + 9
    ref = _run(net, p0, steps, lambda t: "profile")                                       # never a graph
    dev = _run(net, p0, steps, lambda t: "device")
    assert np.array_equal(ref[0], dev[0]) and np.array_equal(ref[1], dev[1])
    assert all(a == b for a, b in zip(ref[2], dev[2]) if not (np.isnan(a) or np.isnan(b)))
    mixed = _run(net, p0, steps, lambda t: ("device", "host", "host", "profile", "device")[(t // 2) % 5])
    assert np.array_equal(ref[0], mixed[0]) and np.array_equal(ref[1], mixed[1])
    host = _run(net, p0, steps, lambda t: "host")
    assert np.array_equal(ref[0], host[0])


def test_set_params_starts_over():
    net = nets()["small"]
    p0 = sy.init_params(net.layers, 0)
    a = _run(net, p0, 25, lambda t: "device", reset_at=12)
    import torch
    from paper_2509_05679_b200 import binding
    ctx = make_ctx(net, p0)
    for t in range(12, 25):
        ctx.step(binding.to_device("fp32", sy.batch_inputs(net, t)), torch.from_numpy(sy.batch_labels(net, t)).cuda())
        ctx.wait_ingest()
    assert np.array_equal(a[0], ctx.params())
    ctx.close()


def test_two_contexts_interleaved():
    import torch
    from paper_2509_05679_b200 import binding
    net = nets()["small"]
    p = [sy.init_params(net.layers, s) for s in (0, 1)]
    alone = [_run(net, q, 15, lambda t: "device")[0] for q in p]
    ctxs = [make_ctx(net, q) for q in p]
    for t in range(15):
        x, y = binding.to_device("fp32", sy.batch_inputs(net, t)), torch.from_numpy(sy.batch_labels(net, t)).cuda()
        for c in ctxs:
            c.step(x, y)
        for c in ctxs:
            c.wait_ingest()
    for c, a in zip(ctxs, alone):
        assert np.array_equal(c.params(), a)
        c.close()


def test_inputs_that_the_ingest_kernel_cannot_read():
    """fdg_step takes any address a copy can read: device buffers that start off the kernel's words and pinned host memory give the
    same weights as aligned device buffers, in kernel-by-kernel iterations and in graphs.  Ordinary host memory is refused before anything is
    enqueued, and the run goes on as if the call had not been made."""
    import torch
    from paper_2509_05679_b200 import binding
    net = nets()["small"]
    p0 = sy.init_params(net.layers, 0)
    steps = 4 * net.K + 9
    ref = _run(net, p0, steps, lambda t: "device")
    ctx = make_ctx(net, p0)
    xraw = torch.empty(net.M * 70 * 4 + 16, dtype=torch.uint8, device="cuda")
    yraw = torch.empty(net.M * 4 + 16, dtype=torch.uint8, device="cuda")
    for t in range(steps):
        x, y = torch.from_numpy(sy.batch_inputs(net, t)), torch.from_numpy(sy.batch_labels(net, t))
        if t % 4 == 0:
            xd, yd = x.cuda(), y.cuda()
        elif t % 4 == 3:
            xd, yd = x.pin_memory(), y.pin_memory()
        else:
            off = (1, 2)[t % 2]
            xd, yd = xraw[off:off + net.M * 70 * 4], yraw[off:off + net.M * 4]
            xd.copy_(x.reshape(-1).view(torch.uint8)); yd.copy_(y.view(torch.uint8))
        torch.cuda.synchronize()
        if t in (0, 2, 20):
            for bad in ((x.numpy(), yd), (xd, y.numpy()), (xd, 1)):
                with pytest.raises(binding.FdgError) as e:
                    ctx.step(*bad)
                assert e.value.status == 1
        ctx.step(xd, yd)
        ctx.wait_ingest()
    assert np.array_equal(ref[0], ctx.params())
    ctx.close()


@pytest.mark.parametrize("serial", [True, False])
@pytest.mark.parametrize("name", ["small", "large"])
def test_host_buffers_filled_by_work_queued_on_the_callers_stream(name, serial):
    """With the caller's streams the host copies are ordered on module 1's stream: a pinned buffer that work queued there is still
    going to fill when fdg_step_host is called gives the weights of buffers that were complete."""
    import torch
    net = nets()[name]
    p0 = sy.init_params(net.layers, 0, bf16=net.dtype == "bf16")
    steps = 2 * net.K + 4
    ref = _run(net, p0, steps, lambda t: "host", serial=serial)
    dt = torch.bfloat16 if net.dtype == "bf16" else torch.float32
    streams = [torch.cuda.Stream() for _ in range(net.K)]
    ctx = make_ctx(net, p0, serial=serial, streams=[s.cuda_stream for s in streams])
    xp = torch.zeros((net.M, net.in_h, net.in_w, net.in_c), dtype=dt).pin_memory()
    yp = torch.zeros(net.M, dtype=torch.int32).pin_memory()
    for t in range(steps):
        xd, yd = torch.from_numpy(sy.batch_inputs(net, t)).to(dt).cuda(), torch.from_numpy(sy.batch_labels(net, t)).cuda()
        torch.cuda.synchronize()
        with torch.cuda.stream(streams[0]):
            torch.cuda._sleep(4_000_000)                    # about 2 ms
            xp.copy_(xd, non_blocking=True)
            yp.copy_(yd, non_blocking=True)
        ctx.step_host(xp, yp)
        ctx.wait_ingest()
    assert np.array_equal(ref[0], ctx.params())
    ctx.close()


def _failing_create():
    """A context whose first large buffer (6 TB) no allocator has: fdg_create fails with FDG_ERR_OOM, through the library's own cudaMalloc."""
    from paper_2509_05679_b200 import binding
    with pytest.raises(binding.FdgError) as e:
        binding.Context(sy.mlp_layers([1 << 18, 10]), [], 1, 1 << 22, 0.05, dtype="bf16", in_shape=(1, 1, 1 << 18), num_classes=10, use_torch_allocator=False)
    assert e.value.status == 5


@pytest.mark.parametrize("fail_at", [2, 5, 8])
def test_a_failed_create_does_not_change_what_other_contexts_compute(fail_at):
    """The CUDA runtime keeps the failed allocation's error for the thread.  The next step of another context on tensor-core linear layers, enqueued
    kernel by kernel (the first with a backward pass) or as a graph, computes the gradients it would have computed without it."""
    import torch
    from paper_2509_05679_b200 import binding
    net = sy.Net("mlp-tc", sy.mlp_layers([256, 256, 256, 10]), [2], 1, 1, 256, 10, 2, 96, 0.05, "bf16")
    p0 = sy.init_params(net.layers, 0, bf16=True)
    steps = fail_at + 1
    ref = _run(net, p0, steps, lambda t: "device")
    ctx = make_ctx(net, p0)
    for t in range(steps):
        if t == fail_at:
            _failing_create()
        x, y = binding.to_device("bf16", sy.batch_inputs(net, t)), torch.from_numpy(sy.batch_labels(net, t)).cuda()
        ctx.step(x, y)
        ctx.wait_ingest()
    assert np.array_equal(ctx.grads(), ref[1]) and np.array_equal(ctx.params(), ref[0])
    ctx.close()


def test_module_times_cover_the_iteration():
    """Every module has a time of its own: one that only pools has no update to end with, and one whose forward pass is a graph of its own counts it.
    A module's time is positive and no longer than its step by the host's clock; in serial mode, where nothing overlaps, all of them together are not."""
    import time
    import torch
    from paper_2509_05679_b200 import binding
    C = 16
    pool = sy.Net("pool-only", [(sy.CONV3X3, 3, C, 1, 1), (sy.RELU, C, C, 1, 0), (sy.MAXPOOL2, C, C, 2, 0), (sy.GLOBAL_AVGPOOL, C, C, 1, 0), (sy.LINEAR, C, 10, 1, 1)],
                  [2, 3], 16, 16, 3, 10, 2, 4, 0.05, "fp32")
    for net, serial in ((pool, False), (pool, True), (nets()["large"], False)):
        ctx = make_ctx(net, sy.init_params(net.layers, 0, bf16=net.dtype == "bf16"), serial=serial)
        x, y = binding.to_device(net.dtype, sy.batch_inputs(net, 0)), torch.from_numpy(sy.batch_labels(net, 0)).cuda()
        for t in range(2 * net.K + 4):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            ctx.step(x, y)
            torch.cuda.synchronize()
            wall = (time.perf_counter() - t0) * 1e3
            ms = ctx.module_times()
            assert np.all(ms > 0) and np.all(ms < wall), (t, ms, wall)
            if serial:
                assert ms.sum() < wall, (t, ms, wall)
        ctx.close()


def test_every_kernel_of_a_step_is_counted():
    """Inputs in device memory cost one kernel more than inputs that are copied in from the host: the one that takes them into the FIFO."""
    import torch
    from paper_2509_05679_b200 import binding
    net = nets()["small"]
    ctx = make_ctx(net, sy.init_params(net.layers, 0))
    x, y = sy.batch_inputs(net, 0), sy.batch_labels(net, 0)
    xd, yd = binding.to_device(net.dtype, x), torch.from_numpy(y).cuda()
    per_step = []
    for step in (lambda: ctx.step(xd, yd), lambda: ctx.step_host(x, y)):
        for _ in range(2 * net.K + 2):
            step()
            ctx.wait_ingest()
        before = ctx.stats()[1]
        step()
        ctx.wait_ingest()
        per_step.append(ctx.stats()[1] - before)
    ctx.close()
    assert per_step[0] == per_step[1] + 1
