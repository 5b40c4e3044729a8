"""Calls of one context on several streams (needs a GB300): a call waits for
its own stream only, whatever the context runs for others, and its kernels keep
to the priority of its stream."""
import json

import numpy as np
import pytest
import torch

from paper_1203_0571_gb300 import binding as B
from paper_1203_0571_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    assert torch.cuda.is_available(), "the gpu tests need a CUDA device"
    return B.Context(0)


def large():
    """A batch of more than 2,048 warps, which runs as two halves where it may,
    and the same for the ragged call's classes."""
    batch = synth.make_workload(0, count=2500)
    b = batch.to("cuda")
    return batch, b, B.make_index(b.offset, b.h, b.w), B.default_opts(max_pix=32 * 32)


@pytest.mark.parametrize("kind", ["fit", "ragged", "host"])
def test_call_does_not_wait_for_another_stream(ctx, kind):
    """Eight batches wait on stream A behind a kernel of about a second; a call
    on stream B ends before that kernel does, with the bytes of a call alone."""
    batch, b, idx, opts = large()
    want = ctx.fit_batch(b.pix, idx, opts=opts)
    outs = [torch.zeros_like(want) for _ in range(9)]
    hpix, hidx = batch.pix.pin_memory(), idx.cpu().pin_memory()
    hout = torch.zeros((batch.count, 64), dtype=torch.uint8).pin_memory()
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    slept = torch.cuda.Event()

    def other():
        if kind == "fit":
            ctx.fit_batch(b.pix, idx, opts=opts, out=outs[8], stream=sb)
        elif kind == "ragged":
            ctx.fit_batch_ragged(b.pix, idx, out=outs[8], stream=sb)
        else:
            ctx.fit_batch_host(hpix, hidx, opts=opts, out=hout, stream=sb)
        sb.synchronize()

    other()                             # first uses (modules, workspaces) are not the subject
    for o in outs:
        o.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(sa):
        torch.cuda._sleep(2_000_000_000)
        slept.record(sa)
        for o in outs[:8]:
            ctx.fit_batch(b.pix, idx, opts=opts, out=o, stream=sa)
    other()
    asleep = not slept.query()
    torch.cuda.synchronize()
    assert asleep, "the call on stream B ended only after the kernel on stream A"
    assert all(torch.equal(o, want) for o in outs[:8])
    if kind == "ragged":                # other tiles and warps per stamp: other sums
        assert torch.equal(outs[8].view(torch.int32)[:, 10], want.view(torch.int32)[:, 10])
    else:
        assert torch.equal(hout.cuda() if kind == "host" else outs[8], want)


def streams_of(call, tmp_path):
    """The streams on which the estimator's kernels of a call run."""
    path = str(tmp_path / "trace.json")
    for _ in range(3):                  # a process's first profile can come back without kernels
        call()
        torch.cuda.synchronize()
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                                torch.profiler.ProfilerActivity.CUDA]) as prof:
            call()
            torch.cuda.synchronize()
        prof.export_chrome_trace(path)
        with open(path) as f:
            ev = json.load(f)["traceEvents"]
        found = {e["args"]["stream"] for e in ev if e.get("cat") == "kernel" and "estimator_kernel" in e["name"]}
        if found:
            return found
    pytest.skip("the profiler records no kernels here")


@pytest.mark.parametrize("kind", ["fit", "ragged"])
def test_kernels_keep_to_the_streams_priority(ctx, kind, tmp_path):
    """The context's own streams have the default priority: a call on a stream
    of another one keeps all of its kernels there."""
    batch, b, idx, opts = large()
    f = ctx.fit_batch if kind == "fit" else ctx.fit_batch_ragged
    out = torch.zeros((batch.count, 64), dtype=torch.uint8, device="cuda")
    high, plain = torch.cuda.Stream(priority=-1), torch.cuda.Stream()
    assert len(streams_of(lambda: f(b.pix, idx, opts=opts, out=out, stream=plain), tmp_path)) > 1
    assert len(streams_of(lambda: f(b.pix, idx, opts=opts, out=out, stream=high), tmp_path)) == 1


def test_call_beside_a_capture(ctx):
    """A call on one stream while the same thread captures another in global
    mode, with the context's side streams in use elsewhere: the capture goes on,
    and the call runs."""
    batch, b, idx, opts = large()
    want = ctx.fit_batch(b.pix, idx, opts=opts)
    outs = [torch.zeros_like(want) for _ in range(2)]
    x = torch.zeros(16, device="cuda")
    sa, sb = torch.cuda.Stream(), torch.cuda.Stream()
    for o, s in zip(outs, (sa, sb)):
        ctx.fit_batch(b.pix, idx, opts=opts, out=o, stream=s)
    torch.cuda.synchronize()
    outs[1].zero_()
    with torch.cuda.stream(sa):
        torch.cuda._sleep(200_000_000)
        ctx.fit_batch(b.pix, idx, opts=opts, out=outs[0], stream=sa)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        x += 1
        ctx.fit_batch(b.pix, idx, opts=opts, out=outs[1], stream=sb)
        x += 1
    torch.cuda.synchronize()
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want)
    graph.replay()
    torch.cuda.synchronize()
    assert float(x[0]) == 2.0
